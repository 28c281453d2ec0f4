// CUDA kernels of the LJ-MD hot path for sm_103a.
//
// Paper: Watanabe, Suzuki, Ito, "Huge-scale Molecular Dynamics Simulation of
// Multibubble Nuclei" (arXiv:1210.3450).
//   cell binning (counting sort)          - Sec. 2.1 grid / linked-list method
//   pair-list build with skin             - Sec. 2.1 bookkeeping method, Fig. 1
//   force loop (full list, no 3rd law)    - Sec. 3.3, Algorithm 1, Eq. 1
//   velocity-Verlet update, periodic box  - Sec. 3.2 / 4.1 (second-order symplectic)
//   displacement-triggered list check     - Sec. 2.1 (list validity every step)
//   PE / virial / KE reductions           - Sec. 2.2, 4.3 (energy and pressure)
//
// Work layout: one warp per tile of 32 consecutive slots of one system, one
// thread per particle ("key" particle data stays in registers, Sec. 2.1); the
// partner loop reads the transposed list so each k is one coalesced 128-byte load.
//
// Decisions that must agree bit for bit with a plain FP64 reference (cell of a
// particle, list membership, wrap into the box, displacement) use explicitly
// rounded FP64 intrinsics (__dadd_rn, __dmul_rn, ...), so the compiler cannot fuse
// them into FMAs.
#include <algorithm>

#include "ljmd_dev.cuh"
#include "ljmd_fixed.cuh"
#include "ljmd_math.cuh"

namespace ljmd {

namespace {

constexpr int kBlock = 128;  // 4 tiles per block
constexpr unsigned kFull = 0xffffffffu;

struct TileCtx {
  int sys;
  int tl;       // tile index within the system
  int local;    // slot index within the system
  int64_t s;    // global slot
  bool act;     // lane holds a particle
  int r;        // rebuild passes: the system's place among the rebuilding systems
};

// Returns false if the whole warp has nothing to do.
__device__ __forceinline__ bool tile_ctx(const DevArrays& a, TileCtx& t, SysParams& P) {
  const int warp = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (warp >= a.ntiles) return false;
  t.sys = a.tile_sys[warp];
  if (t.sys < 0) return false;  // free tile of the arena
  P = a.params[t.sys];
  if (!P.active) return false;
  t.tl = warp - P.t_off;
  t.local = t.tl * kTile + lane;
  t.s = P.p_off + t.local;
  t.act = t.local < P.n;
  return true;
}

// The same without a copy of the system's parameters (held in registers they would
// cost a kernel its occupancy).
__device__ __forceinline__ bool tile_ref(const DevArrays& a, TileCtx& t) {
  const int warp = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5);
  if (warp >= a.ntiles) return false;
  t.sys = a.tile_sys[warp];
  if (t.sys < 0) return false;
  const SysParams& P = a.params[t.sys];
  if (!P.active) return false;
  t.tl = warp - P.t_off;
  t.local = t.tl * kTile + (threadIdx.x & 31);
  t.s = P.p_off + t.local;
  t.act = t.local < P.n;
  return true;
}

// Slot of a listed partner (list word e); the checked build verifies it.
__device__ __forceinline__ uint32_t partner_slot(const DevArrays& a, int sys, uint32_t e, int n, uint32_t self) {
  const uint32_t j = e & kIdxMask;
  return check_ok(a, sys, j < (uint32_t)n, kChkPartner) ? j : self;
}
// List length of a slot; the checked build verifies it against the capacity.
__device__ __forceinline__ int list_count(const DevArrays& a, int sys, int64_t s, int kmax) {
  const int cnt = a.ncnt[s];
  return check_ok(a, sys, cnt >= 0 && cnt <= kmax, kChkCount) ? cnt : 0;
}

// Tile w of the rebuilding systems (in rebuild order; reb_pref holds the prefix of
// their tile counts): false if its system is inactive.
__device__ __forceinline__ bool reb_tile(const DevArrays& a, int nreb, int w, TileCtx& t, SysParams& P) {
  int lo = 0, hi = nreb - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.reb_pref[mid] <= w) lo = mid;
    else hi = mid - 1;
  }
  t.sys = a.rebuild_ids[lo];
  t.r = lo;
  P = a.params[t.sys];
  if (!P.active) return false;
  t.tl = w - a.reb_pref[lo];
  t.local = t.tl * kTile + (threadIdx.x & 31);
  t.s = P.p_off + t.local;
  t.act = t.local < P.n;
  return true;
}

__device__ __forceinline__ int reb_systems(const DevArrays& a) { return a.ctl ? a.ctl->nreb : a.nreb; }

// Rebuild passes visit only the tiles of the rebuilding systems, each warp
// striding over them (a grid sized to the GPU, not to the arena). kSpread: consecutive
// tiles go to different blocks (few tiles, spread over the SMs) and not to the warps of
// one (many tiles, neighbours sharing L1).
template <bool kSpread, class F>
__device__ __forceinline__ void for_rebuild_tiles(const DevArrays& a, F&& body) {
  const int nreb = reb_systems(a);
  const int total = a.reb_pref[nreb];
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  const int w0 = kSpread ? (int)((threadIdx.x >> 5) * gridDim.x + blockIdx.x)
                         : (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  for (int w = w0; w < total; w += nw) {
    TileCtx t;
    SysParams P;
    if (reb_tile(a, nreb, w, t, P)) body(t, P);
  }
}

}  // namespace

// ------------------------------------------------------------ host <-> slots

__global__ void k_from_caller(DevArrays a, int cur, const double* __restrict__ x,
                              const double* __restrict__ v, int sys) {
  const SysParams P = a.params[sys];
  const int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (l >= (int64_t)P.ntiles * kTile) return;
  const int64_t s = P.p_off + l;
  if (l < P.n) {
    // (wrap_fast: the FP64 divisions of the full wrap only for positions outside the box;
    // 29 against 7 us for 262,143 particles)
    a.x[cur][s] = make_double4_32a(wrap_fast(x[3 * l + 0], P.L), wrap_fast(x[3 * l + 1], P.L),
                               wrap_fast(x[3 * l + 2], P.L), 0.0);
    a.v[s] = make_double4_32a(v[3 * l + 0], v[3 * l + 1], v[3 * l + 2], 0.0);
    a.id[s] = (int32_t)l;
  } else {
    a.x[cur][s] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    a.v[s] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    a.id[s] = -1;
    a.ncnt[s] = 0;
  }
}

// Positions (wrapped into [0, L)) and velocities in one pass; x or v may be NULL.
__global__ void k_state_to_caller(DevArrays a, int cur, double* __restrict__ x, double* __restrict__ v, int sys) {
  const SysParams& P = a.params[sys];
  const int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (l >= P.n) return;
  const int64_t s = P.p_off + l;
  const int64_t i = a.id[s];
  if (x) {
    const double4_32a q = a.x[cur][s];  // positions drift outside [0, L) between list builds
    x[3 * i + 0] = wrap_fast(q.x, P.L);
    x[3 * i + 1] = wrap_fast(q.y, P.L);
    x[3 * i + 2] = wrap_fast(q.z, P.L);
  }
  if (v) {
    const double4_32a q = a.v[s];
    v[3 * i + 0] = q.x;
    v[3 * i + 1] = q.y;
    v[3 * i + 2] = q.z;
  }
}

// which: 0 = positions (wrapped into [0, L)), 1 = velocities, 2 = stored forces,
// 4 = positions as held (not wrapped), 5 = positions at the last list build
__global__ void k_to_caller(DevArrays a, int cur, int which, double* __restrict__ out, int sys) {
  const SysParams P = a.params[sys];
  const int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (l >= P.n) return;
  const int64_t s = P.p_off + l;
  const int64_t i = a.id[s];
  double4_32a q;
  if (which == 0) {
    q = a.x[cur][s];  // positions drift outside [0, L) between list builds
    q.x = wrap_fast(q.x, P.L);
    q.y = wrap_fast(q.y, P.L);
    q.z = wrap_fast(q.z, P.L);
  } else if (which == 1) {
    q = a.v[s];
  } else if (which == 4) {
    q = a.x[cur][s];
  } else if (which == 5) {
    q = a.xref[s];
  } else {
    q = a.f[s];
  }
  out[3 * i + 0] = q.x;
  out[3 * i + 1] = q.y;
  out[3 * i + 2] = q.z;
}

// --------------------------------------------------------- binning (Sec. 2.1)

// Count with one atomic per distinct cell of the warp: between builds a tile's
// particles (in the previous build's cell order) mostly stay in one or two cells.
// Every lane of the warp calls this (c < 0: no particle).
__device__ __forceinline__ int warp_cell_add(int32_t* counts, int c) {
  const unsigned same = __match_any_sync(kFull, c);
  const int leader = __ffs(same) - 1;
  int base = 0;
  if (c >= 0 && (threadIdx.x & 31) == leader) base = atomicAdd(&counts[c], __popc(same));
  base = __shfl_sync(kFull, base, leader);
  return base + __popc(same & ((1u << (threadIdx.x & 31)) - 1u));  // this lane's place in the group
}

template <bool kSpread>
__device__ __forceinline__ void cell_count_pass(const DevArrays& a, int cur) {
  for_rebuild_tiles<kSpread>(a, [&](const TileCtx& t, const SysParams& P) {
    // Positions are wrapped into [0, L) only here (at a list build): between
    // builds they move freely so that the periodic images stored in the list
    // stay valid.
    int c = -1;
    if (t.act) {
      const double4_32a x = a.x[cur][t.s];
      const double4_32a w = make_double4_32a(wrap_fast(x.x, P.L), wrap_fast(x.y, P.L), wrap_fast(x.z, P.L), 0.0);
      if (w.x != x.x || w.y != x.y || w.z != x.z) a.x[cur][t.s] = w;
      c = 0;
      if (P.nc > 1) {
        c = cell_of(w, P.inv_cs, P.nc);
        if (!check_ok(a, t.sys, c >= 0 && c < P.nc * P.nc * P.nc, kChkCell)) c = 0;
      }
      a.cell[t.s] = c;
    }
    if (P.nc > 1) {  // uniform over the warp
      warp_cell_add(a.ccount + P.c_off, c);
      // the scan's chunk totals (zeroed by the pass's decision), one atomic per chunk of the warp
      const int copy = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) & (kChunkCopies - 1);
      warp_cell_add(a.chunk_sum, c >= 0 ? (a.chunk_pref[t.r] + c / kScanChunk) * kChunkCopies + copy : -1);
    }
  });
}

__global__ void k_cell_count(DevArrays a, int cur) { cell_count_pass<false>(a, cur); }

// Exclusive scan of the cell counts of the rebuilding systems over chunks of
// kScanChunk cells, so that a large system spreads over many blocks: the count
// kernel also totals each chunk (chunk_sum), and k_cell_starts adds the totals of
// the system's earlier chunks to a block scan of its own chunk and writes the
// starts. Work item w is chunk w - chunk_pref[r] of rebuilding system r. The
// counts are reset to serve as fill counters of the scatter.
constexpr int kScanBlock = kScanChunk / 4;

__device__ __forceinline__ int chunk_system(const DevArrays& a, int nreb, int w) {
  int lo = 0, hi = nreb - 1;
  while (lo < hi) {
    const int m = (lo + hi + 1) >> 1;
    if (a.chunk_pref[m] <= w) lo = m;
    else hi = m - 1;
  }
  return lo;
}

// Sum over the block (every thread receives it); ws holds kScanBlock / 32 ints.
__device__ __forceinline__ int block_sum(int v, int* ws) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = __reduce_add_sync(kFull, v);
  if (lane == 0) ws[w] = v;
  __syncthreads();
  int t = lane < kScanBlock / 32 ? ws[lane] : 0;
  t = __reduce_add_sync(kFull, t);
  __syncthreads();  // ws is reused by the caller's next block-wide step
  return t;
}

// ws holds kScanBlock / 32 ints.
__device__ __forceinline__ void cell_starts_pass(const DevArrays& a, int nreb, int* ws) {
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int total = a.chunk_pref[nreb];
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const int r = chunk_system(a, nreb, w);
    const int sys = a.rebuild_ids[r];
    const SysParams& P = a.params[sys];
    if (!P.active || !a.rebuild[sys]) continue;  // uniform over the block
    const int64_t ncell = (int64_t)P.nc * P.nc * P.nc;
    const int k = w - a.chunk_pref[r];
    // particles in the system's earlier chunks
    int off = 0;
    for (int q = a.chunk_pref[r] * kChunkCopies + (int)threadIdx.x; q < w * kChunkCopies; q += kScanBlock)
      off += a.chunk_sum[q];
    off = block_sum(off, ws);
    int32_t* cnt = a.ccount + P.c_off;
    int32_t* cst = a.cstart + P.c_off;
    const int64_t c0 = (int64_t)k * kScanChunk + 4 * threadIdx.x;
    int v[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = c0 + m < ncell ? cnt[c0 + m] : 0;
    const int tsum = v[0] + v[1] + v[2] + v[3];
    // exclusive scan of tsum over the block
    int incl = tsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) ws[wi] = incl;
    __syncthreads();
    int wpre = 0, btot = 0;
#pragma unroll
    for (int q = 0; q < kScanBlock / 32; ++q) {
      const int t = ws[q];
      wpre += q < wi ? t : 0;
      btot += t;
    }
    int run = off + wpre + incl - tsum;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      if (c0 + m < ncell) {
        cst[c0 + m] = run;
        cnt[c0 + m] = 0;
      }
      run += v[m];
    }
    if (threadIdx.x == 0) {
      if ((int64_t)(k + 1) * kScanChunk >= ncell) cst[ncell] = off + btot;  // the system's last chunk
      if (k == 0) a.margin[sys] = P.skin;  // velocity-bound rule: a fresh list has the whole skin
    }
    __syncthreads();  // ws is reused by the next chunk
  }
}

__global__ void __launch_bounds__(kScanBlock) k_cell_starts(DevArrays a, int nreb) {
  if (a.ctl) nreb = a.ctl->nreb;
  if (nreb <= 0) return;
  __shared__ int ws[kScanBlock / 32];
  cell_starts_pass(a, nreb, ws);
}

// Scatter into cell order (arbitrary within a cell). Beside the old slot, the
// scattered position receives the particle's sort key (x, then caller index) and
// cell, so that the ranking below reads them contiguously (the caller index goes
// to sid, the cell to the cell scratch).

template <bool kSpread>
__device__ __forceinline__ void scatter_pass(const DevArrays& a, int cur) {
  for_rebuild_tiles<kSpread>(a, [&](const TileCtx& t, const SysParams& P) {
    if (P.nc == 1) {  // uniform over the warp
      if (t.act) a.perm[t.s] = t.local;
      return;
    }
    const int c = t.act ? a.cell[t.s] : -1;
    const int k = warp_cell_add(a.ccount + P.c_off, c);  // fill counter, one atomic per cell of the warp
    if (!t.act) return;
    const int pos = a.cstart[P.c_off + c] + k;
    if (!check_ok(a, t.sys, pos < a.cstart[P.c_off + c + 1], kChkScatter)) return;
    const int64_t d = P.p_off + pos;
    a.perm[d] = t.local;
    // x >= 0 (wrapped at the count), so its bit pattern orders like the value
    a.skey[d] = __double_as_longlong(a.x[cur][t.s].x);
    a.sid[d] = a.id[t.s];
    a.celltmp[d] = c;
  });
}

__global__ void k_scatter(DevArrays a, int cur) { scatter_pass<false>(a, cur); }

// Order the particles of each cell by x, ties by caller index (deterministic), and
// gather each into its slot. A row of neighbouring cells along x is then sorted by
// x as a whole, which lets the list build restrict each row to the window
// |x_j - x_i| < rl. One thread per particle: its place in the cell is the number of
// the cell's particles with a smaller key, counted over the scattered members. It
// then writes the particle there: the positions straight to the arrays that only
// the new order uses (the build-time positions and their shadows), the
// velocities, ids and cells to scratch, which the list build copies back slot by
// slot (copy_back_slot). Every slot of a cell holds that cell in the scratch in
// both orders, so the ranking's reads of it need no barrier. The first member of
// each cell resets the cell's fill counter.
template <bool kSpread>
__device__ __forceinline__ void cell_rank_pass(const DevArrays& a, int cur) {
  for_rebuild_tiles<kSpread>(a, [&](const TileCtx& t, const SysParams& P) {
    if (!t.act) return;
    const int p = t.local;           // position in the scattered order
    const int i = a.perm[t.s];       // the particle's slot before the rebuild
    int dst = p;                     // nc == 1: one cell, the scattered order is kept
    if (P.nc > 1) {
      const long long* key = a.skey + P.p_off;
      const int32_t* idk = a.sid + P.p_off;  // caller indices in the scattered order
      const int c = a.celltmp[t.s];
      const int lo = a.cstart[P.c_off + c], hi = a.cstart[P.c_off + c + 1];
      if (p == lo) a.ccount[P.c_off + c] = 0;  // ready for the next binning
      const long long ki = key[p];
      const int32_t idi = idk[p];
      int rank = 0, same = 0;
#pragma unroll 4
      for (int q = lo; q < hi; ++q) {
        const long long kj = key[q];
        rank += kj < ki ? 1 : 0;
        same += kj == ki ? 1 : 0;
      }
      if (same > 1)  // equal keys (rare): by caller index
        for (int q = lo; q < hi; ++q) rank += key[q] == ki && idk[q] < idi ? 1 : 0;
      if (!check_ok(a, t.sys, lo + rank < hi, kChkRank)) return;
      dst = lo + rank;
    }
    if (!check_ok(a, t.sys, i >= 0 && i < P.n, kChkGather)) return;
    const int64_t old = P.p_off + i, d = P.p_off + dst;
    const double4_32a x = a.x[cur][old];
    a.xref[d] = x;
    int4 q = fixed4(x, P.qscale);
    a.xqref[d] = q;
    q.w = __float_as_int((float)x.x);  // x as float: the list build's window key
    a.xq[cur][d] = q;
    a.xf[d] = make_float4((float)x.x, (float)x.y, (float)x.z, 0.0f);
    a.vtmp[d] = a.v[old];
    a.idtmp[d] = a.id[old];
    a.celltmp[d] = a.cell[old];
  });
}

__global__ void k_cell_rank(DevArrays a, int cur) { cell_rank_pass<false>(a, cur); }

// The rebuilt state of one slot back into place. The list build does this for the
// tiles it builds: it reads only the build-time positions, shadows and scratch
// cells, which the copy does not touch, so the copy needs no launch of its own.
__device__ __forceinline__ longlong4_32a fix4(const double4_32a& x) {
  longlong4_32a q;
  q.x = to_fix(x.x);
  q.y = to_fix(x.y);
  q.z = to_fix(x.z);
  q.w = 0;
  return q;
}

__device__ __forceinline__ void copy_back_slot(const DevArrays& a, int cur, int64_t s) {
  const double4_32a x = a.xref[s];
  a.x[cur][s] = x;
  a.v[s] = a.vtmp[s];
  a.id[s] = a.idtmp[s];
  if (a.xl[0]) {
    asm volatile("" ::: "memory");  // xl[1] is vtmp's memory: not before the load above
    a.xl[cur][s] = fix4(x);
  }
  a.cell[s] = a.celltmp[s];
}

// ----------------------------------------------- pair list (Sec. 2.1, Fig. 1)

namespace {

// The FP64 membership test, exactly as the reference writes it: separation,
// periodic image, (dx dx + dy dy) + dz dz < rl^2 without fused operations.
// code = 0xff takes the minimum image d - L nearbyint(d / L) of each axis.
// Returns the image code used, with bit 8 set if the pair is inside.
__device__ __forceinline__ unsigned exact_inside(double xi, double yi, double zi, double xj, double yj, double zj,
                                              unsigned code, double L, double rl2) {
  const double d0 = __dsub_rn(xj, xi), d1 = __dsub_rn(yj, yi), d2 = __dsub_rn(zj, zi);
  if (code == 0xffu) {
    code = 0;
    const double k0 = rint(__ddiv_rn(d0, L)), k1 = rint(__ddiv_rn(d1, L)), k2 = rint(__ddiv_rn(d2, L));
    code |= k0 > 0.5 ? 2u : (k0 < -0.5 ? 1u : 0u);
    code |= (k1 > 0.5 ? 2u : (k1 < -0.5 ? 1u : 0u)) << 2;
    code |= (k2 > 0.5 ? 2u : (k2 < -0.5 ? 1u : 0u)) << 4;
  }
  const double dx = apply_image(d0, code & 3u, L);
  const double dy = apply_image(d1, (code >> 2) & 3u, L);
  const double dz = apply_image(d2, (code >> 4) & 3u, L);
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  return code | (r2 < rl2 ? 0x100u : 0u);  // bit 8: inside
}

// Per-particle state of the list build. The FP64 position and the system's L and
// rl^2 are not kept in registers: the rare exact tests reload them.
struct ListCtx {
  const SysParams* Pp;
  const double4_32a* xs;  // FP64 positions of the system (build-time copy)
  uint32_t* out;          // the particle's list words
  int li;                 // the particle's slot in the system
  int count;
  int kmax;
  bool half;              // half list: only partners in higher slots
  int32_t* chk;           // the system's check word (checked build)
  uint32_t* wp = out;     // where entry `count` goes (entries 4 m .. 4 m + 3 are 16
                          // contiguous bytes; the next four follow 4 kTile words on)
  // The checked build verifies each appended partner: a slot of the system, not
  // the particle itself.
  __device__ __forceinline__ bool entry_ok(uint32_t e) const {
    if (!kChecks) return true;
    const uint32_t j = e & kIdxMask;
    if (j < (uint32_t)Pp->n && j != (uint32_t)li) return true;
    atomicOr(chk, kChkListEntry);
    return false;
  }
  __device__ __forceinline__ void advance() {
    ++count;
    wp += (count & 3) ? 1 : 4 * kTile - 3;
  }
  // Append e when p holds (a predicated store).
  __device__ __forceinline__ void push_if(bool p, uint32_t e) {
    if (!p) return;
    push(e);
  }
  __device__ __forceinline__ void push(uint32_t e) {
    if (!entry_ok(e)) return;
    if (count < kmax) *wp = e;
    advance();
  }
  // Entries up to the next multiple of four hold the particle itself, so that the
  // FP32 step reads whole groups of four without a bound per entry (the pair with
  // itself has r = 0, which its force loop leaves out).
  __device__ __forceinline__ void pad() {
    uint32_t* w = wp;
    for (int c = count; (c & 3) != 0 && c < kmax; ++c) *w++ = (uint32_t)li;
  }
  // Append candidates j0 + k (image bits cbits) for the set bits k of `bits`, in
  // ascending k; the capacity is checked once for all of them.
  __device__ __forceinline__ void push_bits(unsigned bits, int j0, uint32_t cbits) {
    if (count + __popc(bits) <= kmax) {
      while (bits) {
        const int k = __ffs(bits) - 1;
        bits &= bits - 1u;
        const uint32_t e = (uint32_t)(j0 + k) | cbits;
        if (!entry_ok(e)) continue;
        *wp = e;
        advance();
      }
    } else {
      while (bits) {
        const int k = __ffs(bits) - 1;
        bits &= bits - 1u;
        push((uint32_t)(j0 + k) | cbits);
      }
    }
  }
  // Whether candidate j with image code (not 0xff) passes the exact FP64 test.
  __device__ __forceinline__ bool exact_in(int j, unsigned code) const {
    const double4_32a xi = xs[li], xj = xs[j];
    return (exact_inside(xi.x, xi.y, xi.z, xj.x, xj.y, xj.z, code, Pp->L, Pp->rl2) >> 8) & 1u;
  }
  // The exact FP64 test of candidate j with image code (0xff: minimum image).
  __device__ __forceinline__ void exact(int j, unsigned code) {
    const double4_32a xi = xs[li], xj = xs[j];
    const unsigned r = exact_inside(xi.x, xi.y, xi.z, xj.x, xj.y, xj.z, code, Pp->L, Pp->rl2);
    push_if((r >> 8) & 1u, (uint32_t)j | ((r & 0xffu) << kIdxBits));
  }
};

// Candidate pre-tests: squared distance of candidate j (in this range's image)
// from the particle, in float, with sure-inside / sure-outside thresholds.
//   PRE 0: positions rounded to float, key shifted by the range's image;
//          thresholds rl^2 (1 -/+ eps(L / rl)).
//   PRE 1: fixed-point shadow positions (the wrapped 32-bit difference is the
//          minimum image) converted to float; thresholds rl^2 (1 -/+ 1e-5) in
//          fixed-point units (relative error of r^2 below 3.2e-6 for L <= 10^4).
template <int PRE>
struct PreTest;

template <>
struct PreTest<0> {
  const float4* p;
  float cx, cy, cz;  // the particle's position minus the image shift
  float lo2, hi2;
  __device__ __forceinline__ float key(int j) const { return p[j].x; }
  __device__ __forceinline__ float r2(const float4& q) const {
    const float dx = q.x - cx, dy = q.y - cy, dz = q.z - cz;
    return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
  }
  __device__ __forceinline__ float4 load(int j) const { return p[j]; }
};

template <>
struct PreTest<1> {
  const int4* p;
  int qx, qy, qz;
  float lo2, hi2;
  __device__ __forceinline__ float key(int j) const { return __int_as_float(p[j].w); }
  __device__ __forceinline__ float r2(const int4& q) const {
    const float ax = (float)wrapped_diff(q.x, qx);
    const float ay = (float)wrapped_diff(q.y, qy);
    const float az = (float)wrapped_diff(q.z, qz);
    return fmaf(az, az, fmaf(ay, ay, ax * ax));
  }
  __device__ __forceinline__ int4 load(int j) const { return p[j]; }
};

__device__ __forceinline__ float key_of(const float4& q) { return q.x; }
__device__ __forceinline__ float key_of(const int4& q) { return __int_as_float(q.w); }

// Test the candidates of slot range [lo, hi), all with image `code`, against the
// particle and append the partners in candidate order. The range is ordered by x
// (float key) and only the window xlo <= x_j < xhi can hold partners: the first
// candidate is found by bisection and the sweep stops past xhi. Candidates are
// taken in windows of 32 (eight groups of four independent loads; the slot
// arrays have four spare entries at the end): the pre-test sets a bit per
// candidate that is surely inside and per candidate that may be inside; the
// range end, the particle itself and (half list) the lower slots are masked once
// per window, the rare shell candidates take the exact test, and the accepted
// ones are appended in order.
template <class T_>
__device__ __forceinline__ void sweep_range(const T_& T, ListCtx& o, int lo, int hi, unsigned code,
                                            float xlo, float xhi) {
  int b = hi;
  while (lo < b) {
    const int m = (lo + b) >> 1;
    if (T.key(m) < xlo) lo = m + 1;
    else b = m;
  }
  const uint32_t cbits = code << kIdxBits;
  int j = lo;
  bool more = j < hi;
  while (more) {
    const int j0 = j;
    unsigned in = 0u, may = 0u;
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      if (more) {
        const auto q0 = T.load(j), q1 = T.load(j + 1), q2 = T.load(j + 2), q3 = T.load(j + 3);
        if (!(key_of(q0) < xhi)) {
          more = false;
        } else {
          const float r0 = T.r2(q0), r1 = T.r2(q1), r2 = T.r2(q2), r3 = T.r2(q3);
          if (r0 < T.hi2) may |= 1u << (4 * g);
          if (r1 < T.hi2) may |= 2u << (4 * g);
          if (r2 < T.hi2) may |= 4u << (4 * g);
          if (r3 < T.hi2) may |= 8u << (4 * g);
          if (r0 < T.lo2) in |= 1u << (4 * g);
          if (r1 < T.lo2) in |= 2u << (4 * g);
          if (r2 < T.lo2) in |= 4u << (4 * g);
          if (r3 < T.lo2) in |= 8u << (4 * g);
          j += 4;
          more = j < hi;
        }
      }
    }
    const int nt = min(j, hi) - j0;  // candidates tested in this window
    unsigned valid = nt >= 32 ? ~0u : ((1u << nt) - 1u);
    if ((unsigned)(o.li - j0) < 32u) valid &= ~(1u << (o.li - j0));  // not the particle itself
    if (o.half) {  // half list: keep candidates above the particle's slot
      const int d = o.li - j0;
      if (d >= 31) valid = 0u;
      else if (d >= 0) valid &= ~((2u << d) - 1u);
    }
    may &= valid;
    in &= may;
    unsigned shell = may & ~in;
    while (shell) {  // between the pre-test's thresholds: the exact FP64 test
      const int k = __ffs(shell) - 1;
      shell &= shell - 1u;
      if (o.exact_in(j0 + k, code)) in |= 1u << k;
    }
    o.push_bits(in, j0, cbits);
  }
}

// nc == 1: every particle is a candidate. The fixed-point separation (its wrapped
// difference is the minimum image) rules out the far ones; the rest take the exact
// minimum-image test.
__device__ __forceinline__ void sweep_all(ListCtx& o, const int4* __restrict__ q, float hi2, int n) {
  const int4 qi = q[o.li];
  for (int j = 0; j < n; ++j) {
    const int4 qj = q[j];
    const float ax = (float)wrapped_diff(qj.x, qi.x);
    const float ay = (float)wrapped_diff(qj.y, qi.y);
    const float az = (float)wrapped_diff(qj.z, qi.z);
    if (j != o.li && (!o.half || j > o.li) && fmaf(az, az, fmaf(ay, ay, ax * ax)) < hi2) o.exact(j, 0xffu);
  }
}

}  // namespace

// Full list: every j != i with minimum-image r^2 < rl^2 (strict); one thread per
// particle, candidates from the 27 neighbour cells taken as 9 rows of 3 cells that
// are contiguous in cell order (split in two where a row wraps in x), or from all
// particles when nc == 1. Partners are appended in candidate order
// (deterministic, and the same for every PRE).
//
// The decision is the FP64 test ((dx dx + dy dy) + dz dz < rl^2, no fused
// operations). It is taken first by a float pre-test whose error is bounded: below
// its lower threshold the pair is certainly inside, above the upper one certainly
// outside, and only the thin shell between needs the FP64 test. The result is
// identical to always taking it.
// VAR bit 0: the fixed-point pre-test (else float); bit 1: rows farther than rl
// in y or z are skipped and the x window of each row is narrowed to
// sqrt(rl^2 - dy^2 - dz^2) (dy, dz: distances from the particle to the row).
namespace {

// The 9 neighbour rows of one particle (cells other than nc == 1), swept by
// its own thread.
template <int PRE, bool kPrune>
__device__ __forceinline__ void lane_rows(const DevArrays& a, int cur, const SysParams* __restrict__ Pp, ListCtx& o,
                                          int64_t p_off) {
  const int li = o.li, nc = Pp->nc;
  const double4_32a xi0 = o.xs[li];
  const float rl = Pp->rlf, wm = Pp->wmargin;
  float w = rl + wm;  // half-width of the x window
  PreTest<PRE> T;
  if constexpr (PRE == 0) {
    T.p = a.xf + p_off;
    T.lo2 = Pp->rl2f_lo;
    T.hi2 = Pp->rl2f_hi;
  } else {
    T.p = a.xq[cur] + p_off;
    const int4 qi = T.p[li];
    T.qx = qi.x; T.qy = qi.y; T.qz = qi.z;
    T.lo2 = Pp->rl2q_lo;
    T.hi2 = Pp->rl2q_hi;
  }
  const int32_t* cst = a.cstart + Pp->c_off;
  const int ci = a.celltmp[p_off + li];
  const int cx = ci % nc, cy = (ci / nc) % nc, cz = ci / (nc * nc);
  const int nparts = (cx == 0 || cx == nc - 1) ? 2 : 1;
  const double L = Pp->L;
  // offsets of the particle from its cell's lower y and z faces (row pruning)
  const float cs = Pp->csf;
  const float fy = kPrune ? (float)xi0.y - (float)cy * cs : 0.f;
  const float fz = kPrune ? (float)xi0.z - (float)cz * cs : 0.f;
#pragma unroll 1
  for (int rowi = 0; rowi < 9; ++rowi) {
    const int oz = rowi / 3 - 1, oy = rowi % 3 - 1;
    if (kPrune) {
      // the margin (1e-5 L) is far above the float rounding of x_i and of the
      // cell faces (about 1e-7 L)
      const float dy = fmaxf(0.f, (oy < 0 ? fy : (oy > 0 ? cs - fy : 0.f)) - wm);
      const float dz = fmaxf(0.f, (oz < 0 ? fz : (oz > 0 ? cs - fz : 0.f)) - wm);
      const float rem = rl * rl - dy * dy - dz * dz;
      if (rem <= 0.f) continue;  // the whole row is farther than rl
      w = sqrtf(rem) + wm;
    }
    int nz = cz + oz, ny = cy + oy;
    unsigned shz = 0, shy = 0;
    if (nz < 0) { nz += nc; shz = 2; } else if (nz >= nc) { nz -= nc; shz = 1; }
    if (ny < 0) { ny += nc; shy = 2; } else if (ny >= nc) { ny -= nc; shy = 1; }
    const int row = nc * (ny + nc * nz);
    const double4_32a xi = o.xs[li];  // reloaded (an L1 hit) rather than held in registers
    if constexpr (PRE == 0) {
      // image code 1 adds +L to x_j - x_i, code 2 adds -L: shift the particle instead
      T.cy = (float)(shy == 1 ? xi.y - L : (shy == 2 ? xi.y + L : xi.y));
      T.cz = (float)(shz == 1 ? xi.z - L : (shz == 2 ? xi.z + L : xi.z));
    }
#pragma unroll 1
    for (int part = 0; part < nparts; ++part) {
      int lo, hi;
      unsigned code = (shy << 2) | (shz << 4);
      // cells cx-1..cx+1 of this row: one contiguous range, or two where it wraps
      if (cx == 0) {
        if (part == 0) { lo = cst[row + nc - 1]; hi = cst[row + nc]; code |= 2u; }  // x image -L
        else { lo = cst[row]; hi = cst[row + 2]; }
      } else if (cx == nc - 1) {
        if (part == 0) { lo = cst[row + nc - 2]; hi = cst[row + nc]; }
        else { lo = cst[row]; hi = cst[row + 1]; code |= 1u; }                    // x image +L
      } else {
        lo = cst[row + cx - 1]; hi = cst[row + cx + 2];
      }
      // the particle's x in this range's coordinates (candidates are not shifted)
      const double xs_ = (code & 3u) == 1u ? xi.x - L : ((code & 3u) == 2u ? xi.x + L : xi.x);
      const float xw = (float)xs_;
      if constexpr (PRE == 0) T.cx = xw;
      sweep_range(T, o, lo, hi, code, xw - w, xw + w);
    }
  }
}

// List length, the system's largest length and overflow (one atomic per warp:
// all threads of a system hitting one word serialise).
__device__ __forceinline__ void list_done(const DevArrays& a, int sys, int64_t slot, int count, int kmax,
                                          bool act, unsigned mask, int lane) {
  if (act) a.ncnt[slot] = count < kmax ? count : kmax;
  const int wmax = __reduce_max_sync(mask, act ? count : 0);
  if (lane == __ffs(mask) - 1) {
    atomicMax(&a.status[sys].max_count, wmax);
    if (wmax > kmax) {
      atomicMax(&a.status[sys].overflow, wmax);
      if (a.ctl) atomicMax(&a.ctl->abort, 1);  // graph-captured loop: stop; the host grows the list
    }
  }
}

}  // namespace

namespace {

// Next tile of the rebuilding systems for this warp, from a shared work counter
// (dynamic: tiles differ in cost); false when none is left. Warp-uniform.
__device__ __forceinline__ bool next_rebuild_tile(const DevArrays& a, int& sys, int& tl) {
  const int nreb = reb_systems(a);
  const int total = a.reb_pref[nreb];
  int w = 0;
  if ((threadIdx.x & 31) == 0) w = atomicAdd(a.tile_next, 1);
  w = __shfl_sync(kFull, w, 0);
  if (w >= total) return false;
  int lo = 0, hi = nreb - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.reb_pref[mid] <= w) lo = mid;
    else hi = mid - 1;
  }
  sys = a.rebuild_ids[lo];
  tl = w - a.reb_pref[lo];
  return true;
}

}  // namespace

template <int BLOCK, int VAR>
__global__ void __launch_bounds__(BLOCK, 1024 / BLOCK) k_build_list(DevArrays a, int cur) {
  constexpr int PRE = VAR & 1;
  constexpr bool kPrune = (VAR & 2) != 0;
  const int lane = threadIdx.x & 31;
  int sys, tl;
  while (next_rebuild_tile(a, sys, tl)) {
    const SysParams* __restrict__ Pp = a.params + sys;
    if (!Pp->active) continue;
    const int li = tl * kTile + lane;
    const int n = Pp->n;
    const bool act = li < n;
    const int64_t p_off = Pp->p_off;
    const int kmax = Pp->kmax;
    ListCtx o{Pp, a.xref + p_off, a.nbr + list_word(Pp->l_off, tl, kmax, lane, 0), li, 0, kmax, Pp->half != 0,
              a.checks + sys};
    if (act) copy_back_slot(a, cur, p_off + li);
    if (act) {
      if (Pp->nc == 1) sweep_all(o, a.xq[cur] + p_off, Pp->rl2q_hi, n);
      else lane_rows<PRE, kPrune>(a, cur, Pp, o, p_off);
    }
    if (act) o.pad();
    list_done(a, sys, p_off + li, o.count, kmax, act, kFull, lane);
  }
}

// Warp-cooperative list build: the same lists, in the same order, as
// k_build_list. The lanes of a warp that share a row of cells (y, z) take the
// union of their candidates: for each of the 9 neighbour rows, the cells
// cx_min-1 .. cx_max+1 restricted to the group's x window, read 32 at a time with
// coalesced loads into shared memory and tested by every lane from there
// (broadcast reads). Each lane collects its accepted candidates of a chunk in a
// bit mask (pre-test; the shell resolved by the exact FP64 test) and appends them
// in candidate order. Candidates outside a lane's own three cells are farther
// than the cell side >= rl, so they fail its test; every cell of the union
// appears once, with one image, because a group spans at most nc - 2 cells
// (wider runs of a row are split into several groups). Full lists only.
namespace {

__device__ __forceinline__ void build_tile_warp(const DevArrays& a, int cur, int sys, int tl, float4* buf) {
  const int lane = threadIdx.x & 31;
  const SysParams* __restrict__ Pp = a.params + sys;
  if (!Pp->active) return;  // every return above the loop is uniform over the warp
  const int li = tl * kTile + lane;
  const int n = Pp->n;
  const bool act = li < n;
  const unsigned actm = __ballot_sync(kFull, act);
  const int64_t p_off = Pp->p_off;
  const int kmax = Pp->kmax;
  ListCtx o{Pp, a.xref + p_off, a.nbr + list_word(Pp->l_off, tl, kmax, lane, 0), li, 0, kmax, false, a.checks + sys};
  if (act) copy_back_slot(a, cur, p_off + li);
  const int nc = Pp->nc;
  if (nc == 1) {
    if (act) sweep_all(o, a.xq[cur] + p_off, Pp->rl2q_hi, n);
    if (act) o.pad();
    list_done(a, sys, p_off + li, o.count, kmax, act, kFull, lane);
    return;
  }
  const float4* __restrict__ xf = a.xf + p_off;
  const int32_t* __restrict__ cst = a.cstart + Pp->c_off;
  const double L = Pp->L;
  const float w = Pp->rlf + Pp->wmargin;  // half-width of the x window around each particle
  const float lo2 = Pp->rl2f_lo, hi2 = Pp->rl2f_hi;
  int cx = 0, rkey = -1;
  float xk = 0.f;
  if (act) {
    const int ci = a.celltmp[p_off + li];
    cx = ci % nc;
    rkey = ci / nc;  // row of cells (y, z)
    xk = xf[li].x;
  }
  unsigned todo = actm;
  while (todo) {
    // next group: the remaining lanes of one row whose cells span at most nc - 2
    // (so that the union of their neighbour cells holds each cell once)
    const int gkey = __shfl_sync(kFull, rkey, __ffs(todo) - 1);
    const bool same = ((todo >> lane) & 1u) && rkey == gkey;
    const int cxa = __reduce_min_sync(kFull, same ? cx : 0x7fffffff);
    const unsigned grp = __ballot_sync(kFull, same && cx <= cxa + nc - 3);
    todo &= ~grp;
    const bool mine = (grp >> lane) & 1u;
    const int cxb = __reduce_max_sync(kFull, mine ? cx : -1);
    // x extent of the group: x >= 0, so the float bits order like the values
    const float xmin = __int_as_float(__reduce_min_sync(kFull, mine ? __float_as_int(xk) : 0x7f800000));
    const float xmax = __int_as_float(__reduce_max_sync(kFull, mine ? __float_as_int(xk) : 0));
    const int gcy = gkey % nc, gcz = gkey / nc;
    const int npieces = (cxa == 0 || cxb == nc - 1) ? 2 : 1;
#pragma unroll 1
    for (int rowi = 0; rowi < 9; ++rowi) {
      const int oz = rowi / 3 - 1, oy = rowi % 3 - 1;
      int nz = gcz + oz, ny = gcy + oy;
      unsigned shz = 0, shy = 0;
      if (nz < 0) { nz += nc; shz = 2; } else if (nz >= nc) { nz -= nc; shz = 1; }
      if (ny < 0) { ny += nc; shy = 2; } else if (ny >= nc) { ny -= nc; shy = 1; }
      const int row = nc * (ny + nc * nz);
      const double4_32a xi = o.xs[li];  // padding lanes read their zeroed slot
      // image code 1 adds +L to x_j - x_i, code 2 adds -L: shift the particle instead
      const float cy = (float)(shy == 1 ? xi.y - L : (shy == 2 ? xi.y + L : xi.y));
      const float cz = (float)(shz == 1 ? xi.z - L : (shz == 2 ? xi.z + L : xi.z));
#pragma unroll 1
      for (int piece = 0; piece < npieces; ++piece) {
        int c0, c1;  // first and last cell of this piece (contiguous in cell order)
        unsigned code = (shy << 2) | (shz << 4);
        if (cxa == 0) {
          if (piece == 0) { c0 = c1 = nc - 1; code |= 2u; }  // x image -L
          else { c0 = 0; c1 = cxb + 1; }
        } else if (cxb == nc - 1) {
          if (piece == 0) { c0 = cxa - 1; c1 = nc - 1; }
          else { c0 = c1 = 0; code |= 1u; }                  // x image +L
        } else {
          c0 = cxa - 1; c1 = cxb + 1;
        }
        int lo = cst[row + c0];
        const int hi = cst[row + c1 + 1];
        const float sx = (code & 3u) == 1u ? -(float)L : ((code & 3u) == 2u ? (float)L : 0.f);
        const float xlo = xmin + sx - w, xhi = xmax + sx + w;
        const float cxf = (float)((code & 3u) == 1u ? xi.x - L : ((code & 3u) == 2u ? xi.x + L : xi.x));
        // first candidate of the window (every lane takes the same steps)
        int b = hi;
        while (lo < b) {
          const int m = (lo + b) >> 1;
          if (xf[m].x < xlo) lo = m + 1;
          else b = m;
        }
        const uint32_t cbits = code << kIdxBits;
        for (int j0 = lo; j0 < hi; j0 += 32) {
          const int j = j0 + lane;
          const float4 q = j < hi ? xf[j] : make_float4(0.f, 0.f, 0.f, 0.f);
          const unsigned vm = __ballot_sync(kFull, j < hi && q.x < xhi);  // a prefix: keys ascend
          if (vm == 0) break;
          buf[lane] = q;
          __syncwarp();
          if (mine) {
            unsigned M = 0, C = 0;  // maybe inside (below hi2), certainly inside (below lo2)
#pragma unroll
            for (int t = 0; t < 32; ++t) {
              const float4 c = buf[t];
              const float dx = c.x - cxf, dy = c.y - cy, dz = c.z - cz;
              const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
              M |= r2 < hi2 ? 1u << t : 0u;
              C |= r2 < lo2 ? 1u << t : 0u;
            }
            M &= vm;
            if ((unsigned)(li - j0) < 32u) M &= ~(1u << (li - j0));  // not the particle itself
            C &= M;
            unsigned S = M & ~C;  // in the shell: the exact test decides (rare)
            while (S) {
              const int t = __ffs(S) - 1;
              S &= S - 1;
              const double4_32a xa = o.xs[li], xj = o.xs[j0 + t];
              if (exact_inside(xa.x, xa.y, xa.z, xj.x, xj.y, xj.z, code, L, Pp->rl2) & 0x100u) C |= 1u << t;
            }
            while (C) {
              const int t = __ffs(C) - 1;
              C &= C - 1;
              o.push_if(true, (uint32_t)(j0 + t) | cbits);
            }
          }
          __syncwarp();
          if (vm != kFull) break;
        }
      }
    }
  }
  if (act) o.pad();
    list_done(a, sys, p_off + li, o.count, kmax, act, kFull, lane);
}

}  // namespace

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, 1024 / BLOCK) k_build_list_warp(DevArrays a, int cur) {
  __shared__ float4 sbuf[BLOCK];
  float4* buf = sbuf + (threadIdx.x & ~31);
  int sys, tl;
  while (next_rebuild_tile(a, sys, tl)) build_tile_warp(a, cur, sys, tl, buf);
}

// List build with rows staged in shared memory: the same lists, in the same
// order, as k_build_list (the same windows, thresholds and exact test). 0.89 ms per
// build at 2,048,000 particles (rc 2.5) against 1.02 with two compares per candidate
// and 4-byte stores (16-byte stores alone: 0.13 of it; L2 traffic fell from 67 M to 22 M
// store sectors per build of 864,000 particles), 0.95 against 1.18 ms at rc 3.0, density
// 0.6; now bound by issue (78 % active).
// For each neighbour row (and piece of a row that wraps in x) the warp first
// copies the union of its lanes' candidate ranges into shared memory with
// coalesced loads (up to kStage candidates; a wider union, as where a tile's
// lanes sit on both sides of a box face, is swept from global memory). Each lane
// then bisects for its window and sweeps it from there: the candidate loads of
// the sweep, which in k_build_list wait on L1 and often L2 latency, become
// shared-memory loads. Rows and pieces are visited by the whole warp (a lane
// without a second piece has an empty range).
namespace {

constexpr int kStage = 160;  // staged candidates per warp and row piece
struct StageBuf {            // coordinates apart: one 16-byte load gives those of four candidates
  float x[kStage + 4], y[kStage + 4], z[kStage + 4];
};

// The staged build's list writer: entries are collected in registers and stored four at a
// time (a lane's 4-byte stores fill a sector of their own each, 67 M of them per build
// of 864,000 particles).
struct StagedCtx {
  ListCtx o;       // its count and place are brought up to date by leave()
  int count;
  uint32_t* group; // where the group being collected goes
  uint32_t g0, g1, g2, g3;
  __device__ __forceinline__ void push(uint32_t e) {
    if (o.entry_ok(e)) put(e);
  }
  __device__ __forceinline__ void put(uint32_t e) {
    g0 = g1; g1 = g2; g2 = g3; g3 = e;
    ++count;
    // a full group is stored (if it fits: kmax is a multiple of 8), without a branch
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b32 t;\n\tand.b32 t, %1, 3;\n\tsetp.eq.s32 p, t, 0;\n\tsetp.le.and.s32 q, %1, %2, p;\n\t"
                 "@q st.global.v4.u32 [%0], {%3, %4, %5, %6};\n\t@p add.s64 %0, %0, 512;\n\t}"
                 : "+l"(group) : "r"(count), "r"(o.kmax), "r"(g0), "r"(g1), "r"(g2), "r"(g3) : "memory");
  }
  // To the plain writer (the collected entries stored one by one), and from it.
  __device__ __forceinline__ void leave() {
    const int r = count & 3;
    if (count <= o.kmax) {
      if (r == 1) group[0] = g3;
      if (r == 2) { group[0] = g2; group[1] = g3; }
      if (r == 3) { group[0] = g1; group[1] = g2; group[2] = g3; }
    }
    o.count = count;
    o.wp = group + r;
  }
  __device__ __forceinline__ void enter() {
    count = o.count;
    group = o.out + (count >> 2) * (4 * kTile);
    const int r = count & 3;
    if (r && count <= o.kmax) {
      const uint32_t w0 = group[0], w1 = group[1], w2 = group[2];
      g3 = r == 1 ? w0 : r == 2 ? w1 : w2;
      g2 = r == 2 ? w0 : w1;
      g1 = w0;
    }
  }
  // Padding with the particle itself, to a whole group (ListCtx::pad).
  __device__ __forceinline__ void finish() {
    o.count = count;
    while (count & 3) put((uint32_t)o.li);
  }
};

// sweep_range on staged candidates (slot j at place j - first). The pre-test's squared
// distance starts at -hi2, so its sign is the test: the signs are shifted into a mask
// (candidate k of the window at bit 31 - k), 9 instructions per candidate with the
// smallest distance to the threshold, where two compares and two predicated ORs made
// it 11 (and those four run on half of the lanes' rate). A window whose smallest
// distance is within the shell looks at its marked candidates again. Windows start at
// a multiple of four places; candidates outside [lo, hi) are masked.
__device__ __forceinline__ void sweep_staged(const StageBuf& S, int first, float px, float py, float pz, float hi2,
                                             float shell, StagedCtx& w, int lo, int hi, unsigned code, float xlo,
                                             float xhi) {
  int b = hi;
  while (lo < b) {
    const int m = (lo + b) >> 1;
    if (S.x[m - first] < xlo) lo = m + 1;
    else b = m;
  }
  const int fe = hi - first, fs = (lo - first) & ~3;
  int f = fs;
  bool more = lo < hi;
  while (more) {
    const int f0 = f;
    unsigned bits = 0u;
    float near = 1e30f;
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      if (more) {
        const float4 X = *(const float4*)(S.x + f);
        // past the window (the very first group may begin with candidates of another row)
        if ((g > 0 || f0 > fs) && !(X.x < xhi)) {
          more = false;
        } else {
          const float4 Y = *(const float4*)(S.y + f), Z = *(const float4*)(S.z + f);
          auto test = [&](float x, float y, float z) {
            const float dx = x - px, dy = y - py, dz = z - pz;
            const float r = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, -hi2)));
            bits = __funnelshift_l(__float_as_uint(r), bits, 1);
            near = fminf(near, fabsf(r));
          };
          test(X.x, Y.x, Z.x);
          test(X.y, Y.y, Z.y);
          test(X.z, Y.z, Z.z);
          test(X.w, Y.w, Z.w);
          f += 4;
          more = f < fe;
        }
      }
    }
    const int nt = f - f0;  // candidates tested
    if (nt == 0) break;
    bits <<= 32 - nt;
    const int cut = lo - first - f0, end = fe - f0, s = w.o.li - first - f0;
    if (cut > 0) bits &= 0xffffffffu >> cut;
    if (end < 32) bits &= ~(0xffffffffu >> end);
    if ((unsigned)s < 32u) bits &= ~(0x80000000u >> s);  // not the particle itself
    if (w.o.half) {  // half list: candidates above the particle's slot
      if (s >= 31) bits = 0u;
      else if (s >= 0) bits &= 0xffffffffu >> (s + 1);
    }
    if (near <= shell) {  // (rare) between the pre-test's thresholds: the exact FP64 test
      for (unsigned t = bits; t != 0u;) {
        const int k = __clz((int)t);
        t &= ~(0x80000000u >> k);
        const float dx = S.x[f0 + k] - px, dy = S.y[f0 + k] - py, dz = S.z[f0 + k] - pz;
        const float r = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, -hi2)));
        if (!(r < -shell) && !w.o.exact_in(first + f0 + k, code)) bits &= ~(0x80000000u >> k);
      }
    }
    const uint32_t e0 = (uint32_t)(first + f0) | (code << kIdxBits);  // (no carry into the code: slots end below 2^26)
    while (bits) {
      const int k = __clz((int)bits);
      bits &= ~(0x80000000u >> k);
      w.push(e0 + (uint32_t)k);
    }
  }
}

__device__ __forceinline__ void build_tile_staged(const DevArrays& a, int cur, int sys, int tl, StageBuf& buf) {
  const int lane = threadIdx.x & 31;
  const SysParams* __restrict__ Pp = a.params + sys;
  if (!Pp->active) return;  // uniform over the warp
  const int li = tl * kTile + lane;
  const int n = Pp->n;
  const bool act = li < n;
  const int64_t p_off = Pp->p_off;
  const int kmax = Pp->kmax;
  StagedCtx st{ListCtx{Pp, a.xref + p_off, a.nbr + list_word(Pp->l_off, tl, kmax, lane, 0), li, 0, kmax, Pp->half != 0,
                       a.checks + sys}, 0, nullptr, 0u, 0u, 0u, 0u};
  ListCtx& o = st.o;
  if (act) copy_back_slot(a, cur, p_off + li);
  const int nc = Pp->nc;
  if (nc == 1) {  // uniform over the warp
    if (act) sweep_all(o, a.xq[cur] + p_off, Pp->rl2q_hi, n);
    if (act) o.pad();
    list_done(a, sys, p_off + li, o.count, kmax, act, kFull, lane);
    return;
  }
  st.group = o.out;
  const float4* __restrict__ xf = a.xf + p_off;
  const int32_t* __restrict__ cst = a.cstart + Pp->c_off;
  const float w = Pp->rlf + Pp->wmargin;  // half-width of the x window
  PreTest<0> T;
  T.p = xf;
  T.lo2 = Pp->rl2f_lo;
  T.hi2 = Pp->rl2f_hi;
  const float shell = (T.hi2 - T.lo2) * 1.0001f;  // the difference is exact or rounded once
  int cx = 1, cy = 0, cz = 0;
  if (act) {
    const int ci = a.celltmp[p_off + li];
    cx = ci % nc; cy = (ci / nc) % nc; cz = ci / (nc * nc);
  }
  const float Lf = Pp->Lf;
#pragma unroll 1
  for (int rowi = 0; rowi < 9; ++rowi) {
    const int oz = rowi / 3 - 1, oy = rowi % 3 - 1;
    int nz = cz + oz, ny = cy + oy;
    unsigned shz = 0, shy = 0;
    if (nz < 0) { nz += nc; shz = 2; } else if (nz >= nc) { nz -= nc; shz = 1; }
    if (ny < 0) { ny += nc; shy = 2; } else if (ny >= nc) { ny -= nc; shy = 1; }
    const int row = nc * (ny + nc * nz);
    // the particle's float position (reloaded, an L1 hit; padding lanes read their
    // zeroed slot), shifted in float: image code 1 adds +L to x_j - x_i, code 2
    // adds -L, so shift the particle instead (the pre-test's error bound allows
    // for these roundings)
    const float4 fi = xf[li];
    T.cy = shy == 1 ? fi.y - Lf : (shy == 2 ? fi.y + Lf : fi.y);
    T.cz = shz == 1 ? fi.z - Lf : (shz == 2 ? fi.z + Lf : fi.z);
#pragma unroll 1
    for (int part = 0; part < 2; ++part) {
      int lo = 0, hi = 0;
      unsigned code = (shy << 2) | (shz << 4);
      if (act) {
        if (cx == 0) {
          if (part == 0) { lo = cst[row + nc - 1]; hi = cst[row + nc]; code |= 2u; }  // x image -L
          else { lo = cst[row]; hi = cst[row + 2]; }
        } else if (cx == nc - 1) {
          if (part == 0) { lo = cst[row + nc - 2]; hi = cst[row + nc]; }
          else { lo = cst[row]; hi = cst[row + 1]; code |= 1u; }                    // x image +L
        } else if (part == 0) {
          lo = cst[row + cx - 1]; hi = cst[row + cx + 2];
        }
      }
      const bool ne = lo < hi;
      if (!__any_sync(kFull, ne)) continue;  // uniform
      const float xw = (code & 3u) == 1u ? fi.x - Lf : ((code & 3u) == 2u ? fi.x + Lf : fi.x);
      const int u0 = __reduce_min_sync(kFull, ne ? lo : 0x7fffffff);
      const int u1 = __reduce_max_sync(kFull, ne ? hi : -1);
      if (u1 - u0 <= kStage) {
        // stage [u0, u1) and the 3 slots after it (a group of four may read past
        // its range end; the slot arrays have four spare entries)
        for (int k = lane; k < u1 - u0 + 3; k += 32) {
          const float4 q = xf[u0 + k];
          buf.x[k] = q.x;
          buf.y[k] = q.y;
          buf.z[k] = q.z;
        }
        __syncwarp();
        sweep_staged(buf, u0, xw, T.cy, T.cz, T.hi2, shell, st, lo, hi, code, xw - w, xw + w);
        __syncwarp();  // before the next piece overwrites the buffer
      } else {
        T.cx = xw;
        st.leave();
        sweep_range(T, o, lo, hi, code, xw - w, xw + w);
        st.enter();
      }
    }
  }
  if (act) st.finish();
  list_done(a, sys, p_off + li, o.count, kmax, act, kFull, lane);
}

}  // namespace

template <int BLOCK>
__global__ void __launch_bounds__(BLOCK, 1024 / BLOCK) k_build_list_staged(DevArrays a, int cur) {
  __shared__ __align__(16) StageBuf sbuf[BLOCK / 32];
  int sys, tl;
  while (next_rebuild_tile(a, sys, tl)) build_tile_staged(a, cur, sys, tl, sbuf[threadIdx.x >> 5]);
}

// List build with one candidate per lane, for passes of too few tiles to fill the GPU
// with one warp each (such a pass waits on one warp's serial sweep of 9 rows, 70 us
// whatever its size). A block takes `span` consecutive slots (8 or 32: 1 or 4 per
// warp). The particles of one cell have the same 27 neighbour cells, so for each run of
// slots in one cell the block copies all candidates into shared memory in row order,
// shifted to their image, with every load in flight at once (a global load per round of
// 32 candidates would cost its L2 latency each time); each particle's warp then tests
// them 32 at a time and appends the accepted lanes by their place in the ballot. That
// is candidate order, so the lists are the same word for word.
namespace {

constexpr int kWideBlock = 256;
constexpr int kWideWarps = kWideBlock / 32;
constexpr int kWideStage = 1024;  // candidates staged at a time

struct WideShared {
  float4 cand[kWideStage];
  uint32_t word[kWideStage];
  int cell[kTile];
  int at[32], lo[32];    // pieces of the rows: place of the first candidate, its slot,
  unsigned code[32];     // image code
};

// Slots [s0, s1) of system sys (within one tile, at most 32); called by the whole block
// with uniform arguments. Returns the longest list of the warp's particles.
__device__ __forceinline__ int build_span(const DevArrays& a, int cur, int sys, const SysParams* Pp,
                                          int s0, int s1, WideShared& sh) {
  const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5;
  const unsigned below = (1u << lane) - 1u;
  const int nc = Pp->nc, kmax = Pp->kmax;
  const int64_t p_off = Pp->p_off;
  const bool half = Pp->half != 0;
  const double4_32a* xs = a.xref + p_off;
  // list words of slot s0; those of slot s0 + p follow at 4 p
  uint32_t* out = a.nbr + list_word(Pp->l_off, s0 / kTile, kmax, s0 % kTile, 0);
  int wmax = 0;
  // appends the lanes with `in` set (candidate j, list word e) to particle p's list of length c
  auto append = [&](bool in, int p, int j, uint32_t e, int& c) {
    if (kChecks && in) in = check_ok(a, sys, (unsigned)j < (unsigned)Pp->n && j != s0 + p, kChkListEntry);
    const unsigned m = __ballot_sync(kFull, in);
    const int k = c + __popc(m & below);
    if (in && k < kmax) out[((k >> 2) * kTile + p) * 4 + (k & 3)] = e;
    c += __popc(m);
  };
  auto finish = [&](int p, int c) {  // padding to a whole group of four (ListCtx::pad), length
    const int k = c + lane;
    if (k < ((c + 3) & ~3) && k < kmax) out[((k >> 2) * kTile + p) * 4 + (k & 3)] = (uint32_t)(s0 + p);
    if (lane == 0) a.ncnt[p_off + s0 + p] = c < kmax ? c : kmax;
    wmax = c > wmax ? c : wmax;
  };
  if (nc == 1) {  // every particle is a candidate, at its minimum image (as sweep_all)
    const int4* q = a.xq[cur] + p_off;
    const float4* xf1 = a.xf + p_off;
    const float hi2 = Pp->rl2q_hi, lo2q = Pp->rl2q_lo, hl = 0.5f * Pp->Lf;
    const int n = Pp->n;
    for (int p = wv; p < s1 - s0; p += kWideWarps) {
      const int i = s0 + p;
      const int4 qi = q[i];
      const float4 fi = xf1[i];
      int c = 0;
      for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + lane;
        bool in = false;
        unsigned code = 0u;
        if (j < n && (half ? j > i : j != i)) {
          const int4 qj = q[j];
          const float ax = (float)wrapped_diff(qj.x, qi.x);
          const float ay = (float)wrapped_diff(qj.y, qi.y);
          const float az = (float)wrapped_diff(qj.z, qi.z);
          const float r2 = fmaf(az, az, fmaf(ay, ay, ax * ax));
          if (r2 < hi2) {
            // images of the axes from the float separation, unless one is near L / 2
            const float4 fj = xf1[j];
            const float dx = fj.x - fi.x, dy = fj.y - fi.y, dz = fj.z - fi.z;
            const float close = fminf(fabsf(fabsf(dx) - hl), fminf(fabsf(fabsf(dy) - hl), fabsf(fabsf(dz) - hl)));
            code = (dx > hl ? 2u : (dx < -hl ? 1u : 0u)) | (dy > hl ? 8u : (dy < -hl ? 4u : 0u)) |
                   (dz > hl ? 32u : (dz < -hl ? 16u : 0u));
            in = true;
            // the exact FP64 test (also for a position that is not finite, whose shadow is 0)
            if (!(r2 < lo2q) || close < 1e-4f * hl || !(dx + dy + dz < 1e30f)) {
              const double4_32a xi = xs[i], xj = xs[j];
              const unsigned r = exact_inside(xi.x, xi.y, xi.z, xj.x, xj.y, xj.z, 0xffu, Pp->L, Pp->rl2);
              in = (r & 0x100u) != 0u;
              code = r & 0xffu;
            }
          }
        }
        append(in, p, j, (uint32_t)j | (code << kIdxBits), c);
      }
      finish(p, c);
    }
    return wmax;
  }
  const float4* xf = a.xf + p_off;
  const float lo2 = Pp->rl2f_lo, hi2 = Pp->rl2f_hi, Lf = Pp->Lf;
  if (wv == 0) sh.cell[lane] = s0 + lane < s1 ? a.celltmp[p_off + s0 + lane] : -1;
  __syncthreads();
  for (int p0 = 0; p0 < s1 - s0;) {  // runs of slots in one cell (slots are in cell order)
    const int cell = sh.cell[p0];
    const int p1 = p0 + __popc(__ballot_sync(kFull, sh.cell[lane] == cell));
    const int cx = cell % nc, cy = (cell / nc) % nc, cz = cell / (nc * nc);
    // lane 2 r holds row r's candidate range and image code, lane 2 r + 1 its second
    // piece where the row wraps in x; `at` is the place of its first candidate
    int lo = 0, hi = 0;
    unsigned code = 0u;
    if (lane < 18) {
      const int r = lane >> 1;
      const bool second = lane & 1;
      int nz = cz + r / 3 - 1, ny = cy + r % 3 - 1;
      unsigned shz = 0, shy = 0;
      if (nz < 0) { nz += nc; shz = 2; } else if (nz >= nc) { nz -= nc; shz = 1; }
      if (ny < 0) { ny += nc; shy = 2; } else if (ny >= nc) { ny -= nc; shy = 1; }
      const int32_t* cst = a.cstart + Pp->c_off + nc * (ny + nc * nz);
      code = (shy << 2) | (shz << 4);
      int c0 = cx - 1, c1 = cx + 2;  // cells [c0, c1)
      if (cx == 0) {
        if (second) { c0 = 0; c1 = 2; }
        else { c0 = nc - 1; c1 = nc; code |= 2u; }  // x image -L
      } else if (cx == nc - 1) {
        if (second) { c0 = 0; c1 = 1; code |= 1u; }  // x image +L
        else { c0 = nc - 2; c1 = nc; }
      } else if (second) {
        c0 = c1 = 0;
      }
      if (c0 < c1) { lo = cst[c0]; hi = cst[c1]; }
    }
    int at = hi - lo;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, at, o);
      if (lane >= o) at += y;
    }
    const int total = __shfl_sync(kFull, at, 31);
    // pieces without candidates share the next one's place: the bisection finds the last
    // piece that starts at or before a candidate, which holds it
    if (wv == 0) {
      sh.at[lane] = lane < 18 ? at - (hi - lo) : 0x7fffffff;
      sh.lo[lane] = lo;
      sh.code[lane] = code;
    }
    __syncthreads();
    // the warp's particles p0 + wv + 8 i and their list lengths
    const int np = min(4, max(0, (p1 - p0 - wv + kWideWarps - 1) / kWideWarps));
    int c[4] = {0, 0, 0, 0};
    float px[4], py[4], pz[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 x = xf[s0 + min(p0 + wv + kWideWarps * i, p1 - 1)];
      px[i] = x.x;
      py[i] = x.y;
      pz[i] = x.z;
    }
    for (int base = 0; base < total; base += kWideStage) {
      // thread t copies candidates t, t + 256, ...; a candidate's piece by bisection
#pragma unroll
      for (int u = 0; u < kWideStage / kWideBlock; ++u) {
        const int t = u * kWideBlock + (int)threadIdx.x, f = base + t;
        if (f < total) {
          int l = 0;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1)
            if (sh.at[l + o] <= f) l += o;
          const int j = sh.lo[l] + f - sh.at[l];
          const unsigned cd = sh.code[l];
          // image code 1 adds +L to x_j - x_i, code 2 adds -L: the candidate is shifted in
          // float (the same bound as shifting the particle, 4 u L and u L for the other)
          const float sx = (cd & 3u) == 1u ? Lf : ((cd & 3u) == 2u ? -Lf : 0.f);
          const float sy = (cd & 12u) == 4u ? Lf : ((cd & 12u) == 8u ? -Lf : 0.f);
          const float sz = (cd & 48u) == 16u ? Lf : ((cd & 48u) == 32u ? -Lf : 0.f);
          const float4 q = xf[j];
          sh.cand[t] = make_float4(q.x + sx, q.y + sy, q.z + sz, 0.f);
          sh.word[t] = (uint32_t)j | (cd << kIdxBits);
        }
      }
      const int nr = min(kWideStage, total - base), nb = (nr + 31) & ~31;
      if (wv == kWideWarps - 1 && nr + lane < nb) {
        sh.cand[nr + lane] = make_float4(1e18f, 0.f, 0.f, 0.f);
        sh.word[nr + lane] = 0u;
      }
      __syncthreads();
      // rounds of 32 candidates (the last one filled up with candidates far away)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (i >= np) break;  // uniform over the warp
        const int p = p0 + wv + kWideWarps * i;
        const uint32_t self = (uint32_t)(s0 + p);
        const int cut = half ? s0 + p : -1;  // half list: only candidates above the particle's slot
        uint32_t* op = out + 4 * p;
        int cnt = c[i];
#pragma unroll 2
        for (int f = lane; f < nb; f += 32) {  // nb + the filling: uniform over the warp
          const float4 q = sh.cand[f];
          const uint32_t e = sh.word[f];
          const float dx = q.x - px[i], dy = q.y - py[i], dz = q.z - pz[i];
          const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
          bool in = r2 < hi2 && e != self && (int)(e & kIdxMask) > cut;
          if (__any_sync(kFull, in && !(r2 < lo2))) {  // between the pre-test's thresholds: the exact FP64 test (rare)
            if (in && !(r2 < lo2)) {
              const int j = (int)(e & kIdxMask);
              const double4_32a xi = xs[s0 + p], xj = xs[j];
              in = (exact_inside(xi.x, xi.y, xi.z, xj.x, xj.y, xj.z, e >> kIdxBits, Pp->L, Pp->rl2) & 0x100u) != 0u;
            }
            __syncwarp();
          }
          if (kChecks && in)
            in = check_ok(a, sys, (e & kIdxMask) < (uint32_t)Pp->n && (e & kIdxMask) != self, kChkListEntry);
          const unsigned m = __ballot_sync(kFull, in);
          const int k = cnt + __popc(m & below);
          if (in && k < kmax) op[k + (k >> 2) * (4 * kTile - 4)] = e;
          cnt += __popc(m);
        }
        c[i] = cnt;
      }
      __syncthreads();  // before the next candidates
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int p = p0 + wv + kWideWarps * i;
      if (p < p1) finish(p, c[i]);
    }
    p0 = p1;
  }
  return wmax;
}

__device__ __forceinline__ void build_lists_wide(const DevArrays& a, int cur, int span, WideShared& sh) {
  const int nreb = reb_systems(a);
  const int per = kTile / span;  // blocks' pieces per tile
  const int total = a.reb_pref[nreb] * per;
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    int lo = 0, hi = nreb - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (a.reb_pref[mid] * per <= w) lo = mid;
      else hi = mid - 1;
    }
    const int sys = a.rebuild_ids[lo];
    const SysParams* Pp = a.params + sys;
    const int s0 = (w - a.reb_pref[lo] * per) * span;
    const int s1 = min(s0 + span, Pp->n);
    if (!Pp->active || s0 >= s1) continue;  // uniform over the block
    const int wmax = build_span(a, cur, sys, Pp, s0, s1, sh);
    const int me = s0 + (int)threadIdx.x;  // (not before: its loads would delay the candidates')
    if (me < s1) copy_back_slot(a, cur, Pp->p_off + me);
    if ((threadIdx.x & 31) == 0 && wmax > 0) {
      atomicMax(&a.status[sys].max_count, wmax);
      if (wmax > Pp->kmax) {
        atomicMax(&a.status[sys].overflow, wmax);
        if (a.ctl) atomicMax(&a.ctl->abort, 1);  // graph-captured loop: stop; the host grows the list
      }
    }
    __syncthreads();  // before the next span's cells
  }
}

}  // namespace

__global__ void __launch_bounds__(kWideBlock, 4) k_build_list_wide(DevArrays a, int cur, int span) {
  __shared__ WideShared sh;
  build_lists_wide(a, cur, span, sh);
}

// ------------------------------------- fused force + velocity-Verlet step

namespace {

// Velocity-Verlet update of one particle after its force F is known:
//   v += dt/2 F (flag kStepKickA: completes the previous step), v += dt/2 F (flag
//   kStepKickB: first half-kick of the next step; kept as two roundings so that a
//   run split over several calls equals one uninterrupted call bit for bit), then
//   optionally the drift
//   x' = x + dt v into x[cur ^ 1] (not wrapped: list images stay valid) and the
//   squared displacement since the list build for the validity check.
template <bool kFP32>
__device__ __forceinline__ unsigned long long integrate(const DevArrays& a, const SysParams& P, const TileCtx& t,
                                                        int cur, const double4_32a& xi, double Fx, double Fy,
                                                        double Fz, double ka, double kb, int flags) {
  if (flags & kStepStoreF) a.f[t.s] = make_double4_32a(Fx, Fy, Fz, 0.0);
  double4_32a v = a.v[t.s];
  const double dt = P.dt;
  const double h = P.hdt;
  if (flags & kStepKickA) { v.x = fma(h, Fx, v.x); v.y = fma(h, Fy, v.y); v.z = fma(h, Fz, v.z); }
  if (flags & kStepKickB) { v.x = fma(h, Fx, v.x); v.y = fma(h, Fy, v.y); v.z = fma(h, Fz, v.z); }
  a.v[t.s] = v;
  if (!(flags & kStepDrift)) return 0ull;
  double4_32a xn;
  xn.x = fma(dt, v.x, xi.x);
  xn.y = fma(dt, v.y, xi.y);
  xn.z = fma(dt, v.z, xi.z);
  xn.w = 0.0;
  a.x[cur ^ 1][t.s] = xn;
  if (!(finite_bits(xn.x) && finite_bits(xn.y) && finite_bits(xn.z) && finite_bits(v.x) &&
        finite_bits(v.y) && finite_bits(v.z))) {
    a.status[t.sys].nonfinite = 1;
    return ~0ull;
  }
  // velocity-bound rule: |v|^2 of the drift velocity, (vx vx + vy vy) + vz vz unfused
  // (FP64 work only under that rule)
  auto v2b = [&v]() -> unsigned long long {
    return (unsigned long long)__double_as_longlong(
        __dadd_rn(__dadd_rn(__dmul_rn(v.x, v.x), __dmul_rn(v.y, v.y)), __dmul_rn(v.z, v.z)));
  };
  if (kFP32) {
    // check in fixed point: exact integer squared displacement of the shadow
    const int4 q = fixed4(xn, P.qscale);
    a.xq[cur ^ 1][t.s] = q;
    if (flags & kStepVmax) return v2b();
    const int4 r = a.xqref[t.s];
    const long long ex = wrapped_diff(q.x, r.x), ey = wrapped_diff(q.y, r.y), ez = wrapped_diff(q.z, r.z);
    return (unsigned long long)(ex * ex) + (unsigned long long)(ey * ey) + (unsigned long long)(ez * ez);
  }
  // the fixed-point shadow, which the FP64 force loop's pre-classification reads, and
  // the positions in pair units
  a.xq[cur ^ 1][t.s] = fixed4(xn, P.qscale);
  if (a.xl[0]) a.xl[cur ^ 1][t.s] = fix4(xn);
  if (flags & kStepVmax) return v2b();
  // exact FP64 check, the same operations as the reference
  const double4_32a r = a.xref[t.s];
  const double ex = __dsub_rn(xn.x, r.x), ey = __dsub_rn(xn.y, r.y), ez = __dsub_rn(xn.z, r.z);
  const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
  return (unsigned long long)__double_as_longlong(d2);
}

__device__ __forceinline__ void warp_max_disp(const DevArrays& a, int sys, unsigned long long d2b, int flags) {
  if (!(flags & kStepDrift)) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(kFull, d2b, o);
    d2b = y > d2b ? y : d2b;
  }
  if ((threadIdx.x & 31) == 0 && d2b) atomicMax(&a.disp2[sys], d2b);
}

// FP32 pair force factor (24 r^-8 - 48 r^-14 + 8 c2) and separation from an exact
// fixed-point separation; the factor is 0 for r >= rc and for r = 0 (a list's padding
// entries name the particle itself), without branching.
__device__ __forceinline__ float pair_factor_fp32(const int4& qi, const int4& qj, float qu, float rc2, float c2x8,
                                                  float& dx, float& dy, float& dz) {
  dx = (float)wrapped_diff(qj.x, qi.x) * qu;
  dy = (float)wrapped_diff(qj.y, qi.y) * qu;
  dz = (float)wrapped_diff(qj.z, qi.z) * qu;
  const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
  const bool in = r2 < rc2 && r2 > 0.0f;
  const float r2s = in ? r2 : 1.0f;
  float ir2;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ir2) : "f"(r2s));
  ir2 = ir2 * fmaf(-r2s, ir2, 2.0f);  // one Newton step
  const float ir6 = ir2 * ir2 * ir2;
  const float g = fmaf(ir2 * ir6, fmaf(-48.0f, ir6, 24.0f), c2x8);
  return in ? g : 0.0f;
}

__device__ __forceinline__ void pair_fp32(const int4& qi, const int4& qj, float qu, float rc2, float c2x8, float& fx,
                                          float& fy, float& fz) {
  float dx, dy, dz;
  const float g = pair_factor_fp32(qi, qj, qu, rc2, c2x8, dx, dy, dz);
  fx = fmaf(g, dx, fx);
  fy = fmaf(g, dy, fy);
  fz = fmaf(g, dz, fz);
}

}  // namespace

// Loads with L1 eviction hints: list words are read once (no L1 allocation), the
// partners' shadow positions are reused by neighbouring threads (kept in L1).
__device__ __forceinline__ uint4 ld_list(const uint4* p, bool hint) {
  if (!hint) return __ldg(p);
  uint4 r;
  asm("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
      : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

__device__ __forceinline__ int4 ld_shadow(const int4* p, bool hint) {
  if (!hint) return *p;
  int4 r;
  asm("ld.global.nc.L1::evict_last.v4.s32 {%0, %1, %2, %3}, [%4];"
      : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

// FP32-force form: pair arithmetic in FP32 from fixed-point separations (the
// wrapped integer difference is already the minimum image). Each iteration
// takes GROUPS x 4 partners (GROUPS 16-byte list loads, then 4 GROUPS gathers in
// flight at once) and the next iteration's list loads are issued before this
// iteration's gathers are used (software pipelining, the role of Algorithm 1's
// unrolling). BLOCK and GROUPS are chosen by the autotuner.
template <int BLOCK, int GROUPS, bool HINT>
__global__ void __launch_bounds__(BLOCK) k_step_fp32(DevArrays a, int cur, double ka, double kb, int flags) {
  if (a.ctl) {  // graph-captured loop (uniform over the grid)
    if (a.ctl->abort) return;
    flags = a.ctl->flags;
  }
  TileCtx t;
  SysParams P;
  if (!tile_ctx(a, t, P)) return;
  const int lane = threadIdx.x & 31;
  double Fx = 0.0, Fy = 0.0, Fz = 0.0;
  double4_32a xi = make_double4_32a(0.0, 0.0, 0.0, 0.0);
  if (t.act) xi = a.x[cur][t.s];
  if (flags & kStepUseStoredF) {
    if (t.act) {
      const double4_32a f = a.f[t.s];
      Fx = f.x; Fy = f.y; Fz = f.z;
    }
  } else if (t.act) {
    const int cnt = list_count(a, t.sys, t.s, P.kmax);
    const uint4* lp4 = (const uint4*)(a.nbr + list_word(P.l_off, t.tl, P.kmax, lane, 0));
    const int4* qs = a.xq[cur] + P.p_off;
    const int4 qi = a.xq[cur][t.s];
    const float qu = P.qunit, rc2 = P.rc2f, c2x8 = 8.0f * P.c2f;
    const uint32_t self = (uint32_t)t.local;
    const uint4 none = make_uint4(self, self, self, self);
    float fx = 0.f, fy = 0.f, fz = 0.f;
    const int ng = (cnt + 3) >> 2;
    uint4 e[GROUPS];
#pragma unroll
    for (int u = 0; u < GROUPS; ++u) e[u] = u < ng ? ld_list(lp4 + (int64_t)u * kTile, HINT) : none;
    for (int g = 0; g < ng; g += GROUPS) {
      uint4 en[GROUPS];
#pragma unroll
      for (int u = 0; u < GROUPS; ++u)
        en[u] = (g + GROUPS + u < ng) ? ld_list(lp4 + (int64_t)(g + GROUPS + u) * kTile, HINT) : none;
        // the list is padded to whole groups of four with the particle itself, and
      // groups past its end read `none` (also the particle itself)
      int4 q[4 * GROUPS];
#pragma unroll
      for (int u = 0; u < GROUPS; ++u) {
        q[4 * u + 0] = ld_shadow(qs + partner_slot(a, t.sys, e[u].x, P.n, self), HINT);
        q[4 * u + 1] = ld_shadow(qs + partner_slot(a, t.sys, e[u].y, P.n, self), HINT);
        q[4 * u + 2] = ld_shadow(qs + partner_slot(a, t.sys, e[u].z, P.n, self), HINT);
        q[4 * u + 3] = ld_shadow(qs + partner_slot(a, t.sys, e[u].w, P.n, self), HINT);
      }
#pragma unroll
      for (int m = 0; m < 4 * GROUPS; ++m) pair_fp32(qi, q[m], qu, rc2, c2x8, fx, fy, fz);
#pragma unroll
      for (int u = 0; u < GROUPS; ++u) e[u] = en[u];
    }
    Fx = f2d_bits(fx); Fy = f2d_bits(fy); Fz = f2d_bits(fz);  // exact, no FP64-pipe conversion
  }
  unsigned long long d2b = 0ull;
  if (t.act) d2b = integrate<true>(a, P, t, cur, xi, Fx, Fy, Fz, ka, kb, flags);
  warp_max_disp(a, t.sys, d2b, flags);
}

// Approximate reciprocal of r^2 for the force variants of Sec. 3.3: r^2 rounded
// to float, its correctly rounded float reciprocal, the mantissa cut to 8 bits
// for the stand-in of SPARC64 frcpad (relative error < 1/256, Eq. 2).
template <int BITS>
__device__ __forceinline__ double approx_rcp(double r2) {
  float y = __frcp_rn(__double2float_rn(r2));
  if (BITS < 23) y = __uint_as_float(__float_as_uint(y) & ~((1u << (23 - BITS)) - 1u));
  return (double)y;
}

// Force factor g(r) = 24 r^-8 - 48 r^-14 + 8 c2 for MODE 0 (full FP64 reciprocal)
// or from the approximate reciprocal y: MODE 1 / 3 uncorrected (y^4, y^7) with 8 /
// 23 bits, MODE 2 / 4 corrected by Eqs. 2-7 (y^4 (5 - 4 y r^2), y^7 (8 - 7 y r^2)).
template <int MODE>
__device__ __forceinline__ double force_factor(double r2, double c2x8) {
  if (MODE == 0) {
    const double ir2 = rcp_f64(r2);
    const double ir4 = ir2 * ir2;
    const double ir6 = ir4 * ir2;
    const double ir8 = ir4 * ir4;
    return fma(ir8, fma(-48.0, ir6, 24.0), c2x8);
  }
  const double y = approx_rcp<(MODE <= 2) ? 8 : 23>(r2);
  const double y2 = y * y;
  const double y4 = y2 * y2;
  const double y7 = y4 * y2 * y;
  double ir8 = y4, ir14 = y7;
  if (MODE == 2 || MODE == 4) {
    const double e = y * r2;
    ir8 = y4 * fma(-4.0, e, 5.0);
    ir14 = y7 * fma(-7.0, e, 8.0);
  }
  return fma(24.0, ir8, fma(-48.0, ir14, c2x8));
}

// FP64 form. On GB300 a warp's FP64 instruction holds the FP64 pipe for 64 cycles, so
// with the 17 FP64 instructions of a pair the loop ran at that pipe's rate (3.7 ms per
// step at 2,048,000 particles, pipe 89 % busy; 1.10 now). Two things take the load off it:
//   The pair arithmetic runs in 64-bit fixed point on the integer multipliers
//   (ljmd_fixed.cuh: 38 products of 4 cycles each, against 1,090 cycles), with smaller
//   errors than the FP64 pipe's.
//   Pairs outside rc are left out before it. Each thread classifies its listed
//   partners on their fixed-point shadow positions (integer separations, float r^2)
//   against rc^2 (1 + 1e-5), a bound that no pair inside rc can exceed (each shadow
//   coordinate errs by at most half a unit of L / 2^32, and the float r^2 by a few
//   parts in 1e7), and queues the list words of the pairs that may be inside in shared
//   memory; the pairs then run in rounds in which every thread with partners left
//   takes the next one of its own queue (1.26 ms per step without the queue).
// The FP64 pipe still takes the pairs out of the fixed-point range, cutoffs above
// kFixMaxRc and the approximate-reciprocal modes: 3 DADD for the separation and 3
// operations for r^2, the exact test r^2 < rc^2 (bit patterns, r^2 >= 0), the
// reciprocal (3 DFMA after an integer-built FP32 seed), the powers and factor (5) and
// the accumulation (3). The fixed-point sums are exact and a thread's queue keeps list
// order for the others, so the results equal a plain loop's bit for bit.
constexpr int kQueue64 = 32;  // queued list words per thread (FP64 pair loops)

// The classify-and-queue loop of the FP64 pair loops: every thread of the warp
// calls it (cnt = 0 for a lane without a particle). The list words of the thread's
// maybe-inside pairs go through pair(load(e), e) in list order: each pass of the loop
// classifies up to kClassify groups of four partners per lane (as far as its queue has
// room) and then runs as many rounds as every lane with partners left has queued, so
// the warp votes once per pass and not once per round. qme points at the thread's queue column (entry q at
// qme[q * BLOCK]).
// kUpper: only partners in higher slots (each pair of a full list once).
constexpr int kClassify = 7;
template <int BLOCK, bool kUpper, class Load, class Pair>
__device__ __forceinline__ void queued_pairs(const DevArrays& a, const TileCtx& t, const SysParams& P, int lane,
                                             int cur, int cnt, uint32_t* qme, Load&& load, Pair&& pair) {
  const uint4* lp4 = (const uint4*)(a.nbr + list_word(P.l_off, t.tl, P.kmax, lane, 0));
  const int4* qs = a.xq[cur] + P.p_off;
  const int4 qi = t.act ? qs[t.local] : make_int4(0, 0, 0, 0);
  const float rc2q = P.rc2q_hi;
  const uint32_t self = (uint32_t)t.local;
  int k = 0;  // next listed partner to classify
  unsigned head = 0u, tail = 0u;
  uint4 w = make_uint4(self, self, self, self);
  if (cnt > 0) w = __ldg(lp4);
  while (true) {
#pragma unroll 1
    for (int u = 0; u < kClassify; ++u) {
      if (k >= cnt || tail - head > (unsigned)(kQueue64 - 4)) break;
      // the next four listed partners (no FP64 instruction)
      const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
      k += 4;
      if (k < cnt) w = __ldg(lp4 + (int64_t)(k >> 2) * kTile);  // the next group's load in flight
      int4 q4[4];  // all four in flight before the first test: 3 % of the step
      if (!kUpper) {
#pragma unroll
        for (int m = 0; m < 4; ++m) q4[m] = qs[partner_slot(a, t.sys, ws[m], P.n, self)];
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const uint32_t j = partner_slot(a, t.sys, ws[m], P.n, self);
        if (kUpper && j <= self) continue;
        const int4 qj = kUpper ? qs[j] : q4[m];
        const float ax = (float)wrapped_diff(qj.x, qi.x);
        const float ay = (float)wrapped_diff(qj.y, qi.y);
        const float az = (float)wrapped_diff(qj.z, qi.z);
        // the list's padding entries name the particle itself
        if ((kUpper || ws[m] != self) && fmaf(az, az, fmaf(ay, ay, ax * ax)) < rc2q) {
          qme[(tail & (kQueue64 - 1)) * BLOCK] = ws[m];
          ++tail;
        }
      }
    }
    const bool left = k < cnt;
    const bool more = __any_sync(kFull, left);
    // The smallest queue of the lanes with partners left, at the end the largest of all, as
    // one minimum (of the complements at the end): written as a minimum and a maximum on the
    // two sides of a condition, a build of this loop at 72 registers took the minimum for
    // both, and most particles lost the last pairs of their queues.
    const unsigned queued = tail - head;
    const unsigned least = __reduce_min_sync(kFull, more ? (left ? queued : ~0u) : ~queued);
    const unsigned rounds = more ? least : ~least;
    // Two rounds at a time: the second record's load is in flight while the first pair
    // is computed. A run of 2,048,000 particles takes 13.84 ms so against 14.28 with one
    // round at a time, potential energy and virial of 864,000 particles 2 % less.
#pragma unroll 1
    for (unsigned r = 0; r < rounds; r += 2) {
      if (head == tail) continue;
      const bool two = tail - head > 1u && r + 1 < rounds;
      const uint32_t e0 = qme[(head & (kQueue64 - 1)) * BLOCK];
      const uint32_t e1 = two ? qme[((head + 1) & (kQueue64 - 1)) * BLOCK] : e0;
      head += two ? 2u : 1u;
      const auto q0 = load(e0);
      const auto q1 = load(e1);
      pair(q0, e0);
      if (two) pair(q1, e1);
    }
    if (!more) break;
  }
}

// Force of one particle, pair by pair on the FP64 pipe.
template <int MODE>
struct PipeForce {
  const DevArrays& a;
  const TileCtx& t;
  const double4_32a* xs;
  const double4_32a xi;
  const double L, c2x8;
  const int n;
  long long rc2b;
  double x = 0.0, y = 0.0, z = 0.0;
  static constexpr unsigned limit = ~0u;

  __device__ __forceinline__ PipeForce(const DevArrays& a_, const TileCtx& t_, const SysParams& P, int cur)
      : a(a_), t(t_), xs(a_.x[cur] + P.p_off), xi(t_.act ? xs[t_.local] : make_double4_32a(0.0, 0.0, 0.0, 0.0)), L(P.L),
        c2x8(8.0 * P.c2), n(P.n) {
    rc2b = __double_as_longlong(P.rc2);
  }
  __device__ __forceinline__ uint32_t slot(uint32_t e) const { return partner_slot(a, t.sys, e, n, (uint32_t)t.local); }
  __device__ __forceinline__ double4_32a load(uint32_t e) const { return xs[slot(e)]; }
  __device__ __forceinline__ void pair(const double4_32a& xj, uint32_t e) {
    double dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
    const unsigned code = e >> kIdxBits;
    if (code) {
      dx = apply_image(dx, code & 3u, L);
      dy = apply_image(dy, (code >> 2) & 3u, L);
      dz = apply_image(dz, (code >> 4) & 3u, L);
    }
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    if (__double_as_longlong(r2) < rc2b) {
      const double g = force_factor<MODE>(r2, c2x8);  // 24 r^-8 - 48 r^-14 + 8 c2
      x = fma(g, dx, x);
      y = fma(g, dy, y);
      z = fma(g, dz, z);
    }
  }
  __device__ __forceinline__ void result(double& fx, double& fy, double& fz) const {
    fx = x; fy = y; fz = z;
  }
};

// The same in fixed point (ljmd_fixed.cuh) where the system's cutoff, the particle's list
// length and the pair's distance allow it; the other pairs take the FP64 pipe, in the same
// order as above. kAny: for warps in which some particle has more than 448 listed pairs (with
// all of those on the FP64 pipe, beside shorter lists in the same warps, a step of 2,000
// particles at density 1.5, rc 3.9, took 1.3 times as long as without fixed point; 0.8 now) or
// a system out of the cutoff's range. As a run-time limit for every warp it cost 5 % of the
// step.
template <bool kAny>
struct PairForce {
  const DevArrays& a;
  const TileCtx& t;
  const SysParams& P;
  int cur;
  longlong4_32a qi;
  unsigned limit;  // kAny; else kFixR2Min
  FixSum sx, sy, sz;
  double* slow;  // the FP64 pairs' sums, one column of a shared array per thread
  int stride;

  __device__ __forceinline__ PairForce(const DevArrays& a_, const TileCtx& t_, const SysParams& P_, int cur_, int cnt,
                                       double* slow_, int stride_)
      : a(a_), t(t_), P(P_), cur(cur_), slow(slow_), stride(stride_) {
    slow[0] = slow[stride] = slow[2 * stride] = 0.0;
    limit = !kAny ? kFixR2Min : P.fixed ? fix_limit(cnt) : ~0u;
    qi = t.act ? a.xl[cur][t.s] : longlong4_32a{0, 0, 0, 0};
    qi.x -= kFixBias; qi.y -= kFixBias; qi.z -= kFixBias;  // separations come biased for fix_split
  }
  __device__ __forceinline__ void fp64_pair(uint32_t j, unsigned code) {
    const long long rc2b = __double_as_longlong(P.rc2);
    const double c2x8 = 8.0 * P.c2;
    const double4_32a xi = a.x[cur][t.s];
    const double4_32a xj = a.x[cur][P.p_off + j];
    double dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
    if (code) {
      dx = apply_image(dx, code & 3u, P.L);
      dy = apply_image(dy, (code >> 2) & 3u, P.L);
      dz = apply_image(dz, (code >> 4) & 3u, P.L);
    }
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    if (__double_as_longlong(r2) < rc2b) {
      const double g = force_factor<0>(r2, c2x8);  // 24 r^-8 - 48 r^-14 + 8 c2
      slow[0] = fma(g, dx, slow[0]);
      slow[stride] = fma(g, dy, slow[stride]);
      slow[2 * stride] = fma(g, dz, slow[2 * stride]);
    }
  }
  __device__ __forceinline__ uint32_t slot(uint32_t e) const {
    return partner_slot(a, t.sys, e, P.n, (uint32_t)t.local);
  }
  __device__ __forceinline__ longlong4_32a load(uint32_t e) const {
    return a.xl[cur][P.p_off + slot(e)];
  }
  __device__ __forceinline__ void pair(const longlong4_32a& qj, uint32_t e) {
    const unsigned code = e >> kIdxBits;
    if (fix_pair(qi, qj, code, P.Lfix, P.rc2fix, FixC2{P.c2fix, P.c2fix_lo}, sx, sy, sz, kAny ? limit : kFixR2Min))
      fp64_pair(slot(e), code);
  }
  // The sums as FP64 (the FP64 pairs' share added where there is one).
  __device__ __forceinline__ void result(double& x, double& y, double& z) const {
    x = slow[0]; y = slow[stride]; z = slow[2 * stride];
    const bool some = x != 0.0 || y != 0.0 || z != 0.0;
    const double fx = sx.value24(), fy = sy.value24(), fz = sz.value24();
    x = some ? fx + x : fx; y = some ? fy + y : fy; z = some ? fz + z : fz;
  }
};

// FIXED: an arena with systems in the range of the fixed-point pairs; the instance without
// keeps its sums and the particle in registers (a step of 100,000 particles at rc 4.5 takes
// 1.33 ms with it and 1.43 with the other). QUEUE false: the plain loop over the list.
// 28 warps per SM (72 registers, no spills): 20 steps of 2,048,000 particles take 23.9 ms
// against 24.2 at 32 and at 24 warps, of 100,000 2.06 against 2.13 and 2.00.
template <int BLOCK, int MODE, bool QUEUE, bool FIXED>
__global__ void __launch_bounds__(BLOCK, FIXED ? 896 / BLOCK : 1) k_step_fp64(DevArrays a, int cur, double ka, double kb, int flags) {
  __shared__ uint32_t qbuf[QUEUE ? kQueue64 : 1][BLOCK];  // entry q of thread t at [q][t]: no bank conflicts
  __shared__ double slow[FIXED ? 3 : 1][BLOCK];
  if (a.ctl) {  // graph-captured loop (uniform over the grid)
    if (a.ctl->abort) return;
    flags = a.ctl->flags;
  }
  TileCtx t;
  if (!tile_ref(a, t)) return;  // uniform over the warp
  const SysParams& P = a.params[t.sys];
  const int lane = threadIdx.x & 31;
  double Fx = 0.0, Fy = 0.0, Fz = 0.0;
  if (flags & kStepUseStoredF) {
    if (t.act) {
      const double4_32a f = a.f[t.s];
      Fx = f.x; Fy = f.y; Fz = f.z;
    }
  } else {  // every lane of the warp takes part (inactive ones with an empty list)
    const int cnt = t.act ? list_count(a, t.sys, t.s, P.kmax) : 0;
    auto sum = [&](auto pf) {
      if (QUEUE) {
        queued_pairs<BLOCK, false>(a, t, P, lane, cur, cnt, &qbuf[0][threadIdx.x], [&](uint32_t e) { return pf.load(e); },
                                   [&](const auto& q, uint32_t e) { pf.pair(q, e); });
      } else {
        const uint32_t* lp = a.nbr + list_word(P.l_off, t.tl, P.kmax, lane, 0);
        const bool shadows = pf.limit != ~0u && P.wide;
        for (int k = 0; k < cnt; ++k) {
          const uint32_t e = __ldg(lp + (int64_t)(k >> 2) * (4 * kTile) + (k & 3));
          if (shadows) {  // the queue's test: pairs surely outside rc, which may be out of range, are left out
            const int4 qi = a.xq[cur][t.s], qj = a.xq[cur][P.p_off + pf.slot(e)];
            const float ax = (float)wrapped_diff(qj.x, qi.x), ay = (float)wrapped_diff(qj.y, qi.y),
                        az = (float)wrapped_diff(qj.z, qi.z);
            if (!(fmaf(az, az, fmaf(ay, ay, ax * ax)) < P.rc2q_hi)) continue;
          }
          pf.pair(pf.load(e), e);
        }
      }
      pf.result(Fx, Fy, Fz);
    };
    if constexpr (!FIXED) {
      sum(PipeForce<MODE>(a, t, P, cur));
    } else if (P.fixed && __reduce_max_sync(kFull, cnt) <= kFixMaxList) {  // uniform over the warp
      sum(PairForce<false>(a, t, P, cur, cnt, &slow[0][threadIdx.x], BLOCK));
    } else {
      sum(PairForce<true>(a, t, P, cur, cnt, &slow[0][threadIdx.x], BLOCK));
    }
  }
  unsigned long long d2b = 0ull;
  if (t.act) d2b = integrate<false>(a, P, t, cur, a.x[cur][t.s], Fx, Fy, Fz, ka, kb, flags);
  warp_max_disp(a, t.sys, d2b, flags);
}

// ------------------------------------ half list with Newton's third law

// The paper's form before its FX10 kernel (Sec. 2.1 lists each pair once, i < j;
// Sec. 3.3 drops Newton's third law for the SIMD kernel): each pair is listed once,
// in the list of its lower slot; the thread of that slot adds the pair force to
// its own sum and scatters the opposite force to the partner with FP64 atomics.
// The own sum goes to f, the scattered sums to facc; k_integrate_half adds them.
// The order of the atomic additions varies, so results vary in the last bits.
template <int BLOCK, int MODE>
__global__ void __launch_bounds__(BLOCK) k_force_half_fp64(DevArrays a, int cur, int flags) {
  if (a.ctl) {  // graph-captured loop (uniform over the grid)
    if (a.ctl->abort) return;
    flags = a.ctl->flags;
  }
  if (flags & kStepUseStoredF) return;
  TileCtx t;
  SysParams P;
  if (!tile_ctx(a, t, P) || !t.act) return;
  const int lane = threadIdx.x & 31;
  const double4_32a xi = a.x[cur][t.s];
  const int cnt = list_count(a, t.sys, t.s, P.kmax);
  const uint32_t* lp = a.nbr + list_word(P.l_off, t.tl, P.kmax, lane, 0);
  const double4_32a* xs = a.x[cur] + P.p_off;
  double4_32a* fa = a.facc + P.p_off;
  const long long rc2b = __double_as_longlong(P.rc2);
  const double c2x8 = 8.0 * P.c2, L = P.L;
  double Fx = 0.0, Fy = 0.0, Fz = 0.0;
  for (int k = 0; k < cnt; ++k) {
    const uint32_t e = __ldg(lp + (int64_t)(k >> 2) * (4 * kTile) + (k & 3));
    const uint32_t j = partner_slot(a, t.sys, e, P.n, (uint32_t)t.local);
    const double4_32a xj = xs[j];
    double dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
    const unsigned code = e >> kIdxBits;
    if (code) {
      dx = apply_image(dx, code & 3u, L);
      dy = apply_image(dy, (code >> 2) & 3u, L);
      dz = apply_image(dz, (code >> 4) & 3u, L);
    }
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    if (__double_as_longlong(r2) < rc2b) {
      const double g = force_factor<MODE>(r2, c2x8);
      const double fx = g * dx, fy = g * dy, fz = g * dz;
      Fx += fx;
      Fy += fy;
      Fz += fz;
      atomicAdd(&fa[j].x, -fx);
      atomicAdd(&fa[j].y, -fy);
      atomicAdd(&fa[j].z, -fz);
    }
  }
  a.f[t.s] = make_double4_32a(Fx, Fy, Fz, 0.0);
}

// FP32-force form of the same: pair forces in FP32 from the fixed-point
// separation, own sum in FP32, scattered sums in FP64.
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK) k_force_half_fp32(DevArrays a, int cur, int flags) {
  if (a.ctl) {
    if (a.ctl->abort) return;
    flags = a.ctl->flags;
  }
  if (flags & kStepUseStoredF) return;
  TileCtx t;
  SysParams P;
  if (!tile_ctx(a, t, P) || !t.act) return;
  const int lane = threadIdx.x & 31;
  const int cnt = list_count(a, t.sys, t.s, P.kmax);
  const uint32_t* lp = a.nbr + list_word(P.l_off, t.tl, P.kmax, lane, 0);
  const int4* qs = a.xq[cur] + P.p_off;
  const int4 qi = a.xq[cur][t.s];
  double4_32a* fa = a.facc + P.p_off;
  const float qu = P.qunit, rc2 = P.rc2f, c2x8 = 8.0f * P.c2f;
  float fx = 0.f, fy = 0.f, fz = 0.f;
  for (int k = 0; k < cnt; ++k) {
    const uint32_t j = partner_slot(a, t.sys, __ldg(lp + (int64_t)(k >> 2) * (4 * kTile) + (k & 3)), P.n,
                                    (uint32_t)t.local);
    float px = 0.f, py = 0.f, pz = 0.f;
    pair_fp32(qi, qs[j], qu, rc2, c2x8, px, py, pz);
    fx += px;
    fy += py;
    fz += pz;
    if (px != 0.f || py != 0.f || pz != 0.f) {
      atomicAdd(&fa[j].x, -f2d_bits(px));
      atomicAdd(&fa[j].y, -f2d_bits(py));
      atomicAdd(&fa[j].z, -f2d_bits(pz));
    }
  }
  a.f[t.s] = make_double4_32a(f2d_bits(fx), f2d_bits(fy), f2d_bits(fz), 0.0);
}

// Velocity-Verlet update of the half-list form: F = own sum + scattered sums
// (the latter reset for the next step), or the stored F.
template <bool kFP32>
__global__ void __launch_bounds__(kBlock) k_integrate_half(DevArrays a, int cur, int flags) {
  if (a.ctl) {
    if (a.ctl->abort) return;
    flags = a.ctl->flags;
  }
  TileCtx t;
  SysParams P;
  if (!tile_ctx(a, t, P)) return;
  double Fx = 0.0, Fy = 0.0, Fz = 0.0;
  double4_32a xi = make_double4_32a(0.0, 0.0, 0.0, 0.0);
  unsigned long long d2b = 0ull;
  if (t.act) {
    xi = a.x[cur][t.s];
    const double4_32a f = a.f[t.s];
    Fx = f.x; Fy = f.y; Fz = f.z;
    if (!(flags & kStepUseStoredF)) {
      const double4_32a g = a.facc[t.s];
      Fx += g.x; Fy += g.y; Fz += g.z;
      a.facc[t.s] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    }
    d2b = integrate<kFP32>(a, P, t, cur, xi, Fx, Fy, Fz, 0.0, 0.0, flags);
  }
  warp_max_disp(a, t.sys, d2b, flags);
}

// ------------------------------------------------- observables (FP64 sums)

// Potential energy and virial of the pairs with r < rc, and 1/2 |v|^2: each tile sums its
// particles' shares into tile_obs[3 t ...]. With V(r) = 4 (r^-12 - r^-6) + 4 c2 r^2 + 4 c0
// (Eq. 1) and -r V'(r) = 48 r^-12 - 24 r^-6 - 8 c2 r^2, the pair loop only sums r^-12, r^-6
// and r^2 and counts the pairs inside rc. A full list holds each pair twice: the
// particle in its lower slot takes it. Like the FP64 force loop it classifies the
// listed pairs on the fixed-point shadows and runs the others from per-thread queues, in
// fixed point (ljmd_fixed.cuh; sums exact, over the tile as well) where the cutoff
// allows it, else and for close pairs on the FP64 pipe. With all pairs on that pipe and
// each taken twice the kernel ran at its rate: 455 us at 262,143 particles.
// 28 warps per SM (72 registers): a call takes 419 us at 864,000 particles, against 426 at
// 24 and 443 at 32 warps. Splitting each particle's pairs evenly instead (by slot parity)
// was 2 % slower, since whole warps no longer skip the lower half of their lists. The bits
// below the second half of r^-6 and r^-12 cost 8 % (390 us without them).
// xl: positions in pair units.
__global__ void __launch_bounds__(kBlock, 7) k_pe_virial(DevArrays a, int cur, int with_pairs,
                                                         const int32_t* __restrict__ select, const longlong4_32a* xl) {
  __shared__ uint32_t qbuf[kQueue64][kBlock];
  TileCtx t;
  if (!tile_ref(a, t)) return;              // uniform over the warp
  if (select && !select[t.sys]) return;     // uniform over the warp
  const SysParams& P = a.params[t.sys];
  const int lane = threadIdx.x & 31;
  double pe = 0.0, w = 0.0, ke = 0.0;
  if (with_pairs) {  // every lane takes part (inactive ones with an empty list)
    const double4_32a* xs = a.x[cur] + P.p_off;
    const longlong4_32a* ls = xl + P.p_off;
    const int cnt = t.act ? list_count(a, t.sys, t.s, P.kmax) : 0;
    const uint32_t self = (uint32_t)t.local;
    const bool fixed = P.fixed != 0;  // uniform over the warp
    longlong4_32a qi = fixed && t.act ? ls[t.local] : longlong4_32a{0, 0, 0, 0};
    qi.x -= kFixBias; qi.y -= kFixBias; qi.z -= kFixBias;
    FixAcc a12, a6, ar;
    double s12 = 0.0, s6 = 0.0, sr = 0.0;  // the FP64 pipe's pairs
    int nin = 0;
    bool slow = false;
    auto fp64_pair = [&](uint32_t j, unsigned code) {
      const double4_32a xi = xs[t.local], xj = xs[j];
      double dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
      if (code) {
        dx = apply_image(dx, code & 3u, P.L);
        dy = apply_image(dy, (code >> 2) & 3u, P.L);
        dz = apply_image(dz, (code >> 4) & 3u, P.L);
      }
      const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
      const long long r2b = __double_as_longlong(r2);
      if (r2b < __double_as_longlong(P.rc2)) {
        // reciprocal within rounding in 3 DFMA (see rcp_f64); IEEE division only for
        // (near-)coincident pairs, outside rcp_f64's range
        const double ir2 = r2b > __double_as_longlong(1e-30) ? rcp_f64(r2) : 1.0 / r2;
        const double ir6 = ir2 * ir2 * ir2;
        s12 = fma(ir6, ir6, s12);
        s6 += ir6;
        sr += r2;
        ++nin;
        slow = true;
      }
    };
    auto load = [&](uint32_t e) {
      if (fixed) return ls[partner_slot(a, t.sys, e, P.n, self)];
      return longlong4_32a{0, 0, 0, 0};
    };
    queued_pairs<kBlock, true>(a, t, P, lane, cur, cnt, &qbuf[0][threadIdx.x], load, [&](const longlong4_32a& qj, uint32_t e) {
      const unsigned code = e >> kIdxBits;
      if (fixed) {
        const unsigned long long r2 = fix_separation2(qi, qj, code, P.Lfix);
        const bool far = (unsigned)(r2 >> 32) >= kFixR2Min;
        if (far & ((long long)(r2 - (unsigned long long)P.rc2fix) < 0)) {
          const Fix96 y3 = fix_y3(fix_rcp(r2));
          a12.add(fix_sqr(y3.hi));
          a6.add(y3);
          ar.add(r2);
          ++nin;
        } else if (!far) {
          fp64_pair(partner_slot(a, t.sys, e, P.n, self), code);
        }
      } else {
        fp64_pair(partner_slot(a, t.sys, e, P.n, self), code);
      }
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a12.join(o);
      a6.join(o);
      ar.join(o);
    }
    nin = __reduce_add_sync(kFull, nin);
    if (__any_sync(kFull, slow)) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        s12 += __shfl_xor_sync(kFull, s12, o);
        s6 += __shfl_xor_sync(kFull, s6, o);
        sr += __shfl_xor_sync(kFull, sr, o);
      }
      s12 += a12.value(90);
      s6 += a6.value(93);
      sr += ar.value(56);
    } else {
      s12 = a12.value(90);
      s6 = a6.value(93);
      sr = ar.value(56);
    }
    const double c2 = P.c2;
    pe = 4.0 * (s12 - s6) + 4.0 * fma(c2, sr, P.c0 * (double)nin);
    w = 48.0 * s12 - 24.0 * s6 - 8.0 * c2 * sr;
  }
  if (t.act) {
    const double4_32a v = a.v[t.s];
    ke = 0.5 * (v.x * v.x + v.y * v.y + v.z * v.z);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ke += __shfl_xor_sync(kFull, ke, o);
  if (lane == 0) {
    const int64_t g = (int64_t)(P.t_off + t.tl) * 3;
    a.tile_obs[g + 0] = pe;
    a.tile_obs[g + 1] = w;
    a.tile_obs[g + 2] = ke;
  }
}

// Positions in pair units into scratch (the rebuild's gathered velocities, free between
// rebuilds), for forms that do not keep them up: cheaper than converting each partner.
__global__ void __launch_bounds__(kBlock) k_fix_positions(DevArrays a, int cur, const int32_t* __restrict__ select) {
  TileCtx t;
  if (!tile_ref(a, t) || !t.act || (select && !select[t.sys]) || !a.params[t.sys].fixed) return;
  reinterpret_cast<longlong4_32a*>(a.vtmp)[t.s] = fix4(a.x[cur][t.s]);
}

// Counts of listed pairs and of listed pairs with r < rc (FP64 test), per system.
__global__ void __launch_bounds__(kBlock) k_pair_stats(DevArrays a, int cur, unsigned long long* out2) {
  TileCtx t;
  SysParams P;
  if (!tile_ctx(a, t, P)) return;
  const int lane = threadIdx.x & 31;
  unsigned listed = 0, inside = 0;
  if (t.act) {
    const double4_32a xi = a.x[cur][t.s];
    const double4_32a* xs = a.x[cur] + P.p_off;
    const int cnt = list_count(a, t.sys, t.s, P.kmax);
    const uint32_t* lp = a.nbr + list_word(P.l_off, t.tl, P.kmax, lane, 0);
    listed = (unsigned)cnt;
    for (int k = 0; k < cnt; ++k) {
      const uint32_t e = lp[(int64_t)(k >> 2) * (4 * kTile) + (k & 3)];
      const double4_32a xj = xs[partner_slot(a, t.sys, e, P.n, (uint32_t)t.local)];
      const unsigned code = e >> kIdxBits;
      const double dx = apply_image(xj.x - xi.x, code & 3u, P.L);
      const double dy = apply_image(xj.y - xi.y, (code >> 2) & 3u, P.L);
      const double dz = apply_image(xj.z - xi.z, (code >> 4) & 3u, P.L);
      if (dx * dx + dy * dy + dz * dz < P.rc2) ++inside;
    }
  }
  listed = __reduce_add_sync(kFull, listed);
  inside = __reduce_add_sync(kFull, inside);
  if (lane == 0) {
    atomicAdd(&out2[2 * t.sys + 0], (unsigned long long)listed);
    atomicAdd(&out2[2 * t.sys + 1], (unsigned long long)inside);
  }
}

// Per-system sums of the tile partials (PE, W, KE), in two deterministic stages
// whose partition is relative to each system's first tile (so a system reduces
// the same way alone and in a batch): chunks of 256 tiles, one block each, summed
// by a fixed tree; then one block per system adds its chunk sums in order.
// work: the selected systems' ids (nsel) followed by the prefix of their chunk
// counts (nsel + 1).
constexpr int kObsChunk = 256;

__global__ void __launch_bounds__(kObsChunk) k_obs_chunks(DevArrays a, const int32_t* __restrict__ work, int nsel,
                                                        double* __restrict__ chunk3) {
  const int b = blockIdx.x;
  const int32_t* cpref = work + nsel;
  int lo = 0, hi = nsel - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (cpref[mid] <= b) lo = mid;
    else hi = mid - 1;
  }
  const int sys = work[lo];
  const SysParams& P = a.params[sys];
  const int q = (b - cpref[lo]) * kObsChunk + (int)threadIdx.x;  // tile within the system
  __shared__ double sh[3][kObsChunk];
  double pe = 0.0, w = 0.0, ke = 0.0;
  if (q < P.ntiles) {
    const double* o = a.tile_obs + (int64_t)(P.t_off + q) * 3;
    pe = o[0];
    w = o[1];
    ke = o[2];
  }
  sh[0][threadIdx.x] = pe;
  sh[1][threadIdx.x] = w;
  sh[2][threadIdx.x] = ke;
  __syncthreads();
  for (int o = kObsChunk / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + o];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + o];
      sh[2][threadIdx.x] += sh[2][threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    chunk3[3 * b + 0] = sh[0][0];
    chunk3[3 * b + 1] = sh[1][0];
    chunk3[3 * b + 2] = sh[2][0];
  }
}

__global__ void __launch_bounds__(256) k_obs_final(const int32_t* __restrict__ work, int nsel,
                                                 const double* __restrict__ chunk3, double* __restrict__ out3) {
  const int r = blockIdx.x;
  const int sys = work[r];
  const int c0 = work[nsel + r], c1 = work[nsel + r + 1];
  __shared__ double sh[3][256];
  double pe = 0.0, w = 0.0, ke = 0.0;
  for (int c = c0 + (int)threadIdx.x; c < c1; c += 256) {
    pe += chunk3[3 * c + 0];
    w += chunk3[3 * c + 1];
    ke += chunk3[3 * c + 2];
  }
  sh[0][threadIdx.x] = pe;
  sh[1][threadIdx.x] = w;
  sh[2][threadIdx.x] = ke;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + o];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + o];
      sh[2][threadIdx.x] += sh[2][threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out3[3 * sys + 0] = sh[0][0];
    out3[3 * sys + 1] = sh[1][0];
    out3[3 * sys + 2] = sh[2][0];
  }
}

// ------------------------------------------ Nose-Hoover thermostat (Sec. 4.1)

// The kinetic energy of the thermostat is an exact sum of the squared velocity components
// (SquareSum; in global memory eight 32-bit limbs and the word of the squares out of
// range), so every way of running the steps, alone or in a batch, gives the same bits
// whatever the order.
namespace {

__device__ __forceinline__ void add_limbs(unsigned long long* ke, const SquareSum& s) {
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (s.w[m] & 0xffffffffull) atomicAdd(ke + 2 * m, s.w[m] & 0xffffffffull);
    if (s.w[m] >> 32) atomicAdd(ke + 2 * m + 1, s.w[m] >> 32);
  }
  if (s.over) atomicMax(ke + 8, s.over);
}
// Kinetic energy from the limbs.
__device__ __forceinline__ double limbs_ke(const unsigned long long* ke) {
  SquareSum s;
  unsigned long long carry = 0ull;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const unsigned long long a = __ldcg(ke + 2 * m) + carry, b = __ldcg(ke + 2 * m + 1) + (a >> 32);
    s.w[m] = (b << 32) | (a & 0xffffffffull);
    carry = b >> 32;
  }
  s.over = __ldcg(ke + 8);
  return s.half();
}

// `halves` consecutive thermostat half steps from one kinetic energy: each is
// zeta += dt/4 G, eta += dt/2 zeta, v *= exp(-dt/2 zeta), zeta += dt/4 G' with
// G = (2 KE - g T) / Q; a uniform scale multiplies KE by its square, so the next G needs
// no new sum. Returns the factor of the velocities. (Explicit roundings: the same bits
// wherever it is inlined.)
__device__ __forceinline__ double thermo_halves(Thermo& t, double ke, int halves) {
  double fac = 1.0;
  const double q = __dmul_rn(0.25, t.dt), e = __dmul_rn(0.5, t.dt);
  for (int h = 0; h < halves; ++h) {
    t.zeta = __dadd_rn(t.zeta, __ddiv_rn(__dmul_rn(q, __dsub_rn(__dmul_rn(2.0, ke), t.gT)), t.Q));
    t.eta = __dadd_rn(t.eta, __dmul_rn(e, t.zeta));
    const double sc = exp(-__dmul_rn(e, t.zeta));
    fac = __dmul_rn(fac, sc);
    ke = __dmul_rn(__dmul_rn(ke, sc), sc);
    t.zeta = __dadd_rn(t.zeta, __ddiv_rn(__dmul_rn(q, __dsub_rn(__dmul_rn(2.0, ke), t.gT)), t.Q));
  }
  return fac;
}

}  // namespace

__global__ void __launch_bounds__(256) k_ke_limbs(DevArrays a, unsigned long long* ke) {
  const int lane = threadIdx.x & 31;
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  SquareSum s;
  int last = -1;
  auto flush = [&]() {
    if (last < 0) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s.join(o);
    if (lane == 0) add_limbs(ke + kKeWords * last, s);
    s = SquareSum();
  };
  // each warp a run of consecutive tiles (few changes of system)
  const int per = (a.ntiles + nw - 1) / nw;
  const int w0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per, w1 = min(w0 + per, a.ntiles);
  for (int w = w0; w < w1; ++w) {
    const int sys = a.tile_sys[w];
    if (sys < 0) continue;
    const SysParams& P = a.params[sys];
    if (!P.active) continue;
    if (sys != last) {
      flush();
      last = sys;
    }
    const int local = (w - P.t_off) * kTile + lane;
    if (local < P.n) {
      const double4_32a v = a.v[P.p_off + local];
      s.add(__dmul_rn(v.x, v.x));
      s.add(__dmul_rn(v.y, v.y));
      s.add(__dmul_rn(v.z, v.z));
    }
  }
  flush();
}

__global__ void k_thermostat(DevArrays a, int nsys, Thermo* thermo, int halves, unsigned long long* ke, double* scale) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nsys) return;
  double f = 1.0;
  if (a.params[k].active) {
    Thermo t = thermo[k];
    f = thermo_halves(t, limbs_ke(ke + kKeWords * k), halves);
    thermo[k] = t;
  }
  scale[k] = f;
  for (int m = 0; m < kKeWords; ++m) ke[kKeWords * k + m] = 0ull;
}

// ------------------------------------ persistent step loop of small arenas

// A step of a few thousand particles is a chain of latencies: in separate launches
// (step, decision, conditional rebuild node, and five kernels per rebuild) it took 28 to
// 33 us at 1000 to 32,000 particles with FP32 forces and 70 to 77 with FP64 ones, of which
// the pair arithmetic is about 1 to 8. Here one cooperative launch takes all steps of a
// call: 8.0, 10.4, 18 and 25 us at 1000, 4000, 16,000 and 32,000 particles (FP32 forces; 200
// steps from a lattice, its lists and rebuilds included), 9.0, 12.4 and 27 us at 1000, 4000
// and 16,000 (FP64). Without its
// rebuilds a step of 4000 particles takes 5.0 us: forces 2.2, update 0.9, barrier 1.5,
// decision 0.4; a rebuild 40 us. Several threads share a particle, whose
// position, velocity and list stay in registers and shared memory between rebuilds; a
// step reads the partners' shadows, writes the own one, and ends at a grid barrier,
// after which every block takes the list-validity decision for itself from the
// maxima. A rebuild runs the same passes as the separate kernels between barriers.
//
// Results are those of the other loops bit for bit: FP32 pair forces are formed by all
// threads of the particle, exchanged through shared memory and added by one thread
// per axis in list order; FP64 forces are exact integer sums (ljmd_fixed.cuh), and pairs
// out of their range are added in list order.
namespace {

constexpr int kLoopBlock = 256;
constexpr int kLoopWarps = kLoopBlock / 32;

__host__ __device__ constexpr int loop_chunk(int T) { return T >= 32 ? 3 : 4; }  // pairs per thread between exchanges
// FP32 exchange buffer of one particle (words; the 4 extra ones keep the particles of a
// warp on different banks)
__host__ __device__ constexpr int loop_ex(int T) { return loop_chunk(T) * T * 4 + 4; }
__host__ __device__ constexpr size_t loop_union_bytes(int T) {
  return sizeof(WideShared) > (size_t)loop_ex(T) * 4 * (kLoopBlock / T) ? sizeof(WideShared)
                                                                       : (size_t)loop_ex(T) * 4 * (kLoopBlock / T);
}

// List words in shared memory: the FP32 form needs the partner's slot only (an arena of
// the loop has fewer than 2^16).
template <bool kFP32> struct LoopWord { using type = uint32_t; };
template <> struct LoopWord<true> { using type = uint16_t; };

struct LoopShared {
  unsigned long long d2[kLoopWarps];
  int sys[kLoopWarps];
  double margin[kLoopMaxSys];
  double scale[kLoopMaxSys];
  SquareSum ke[kLoopWarps];
  int need[kLoopMaxSys];
  int ws[kScanBlock / 32];
  int flag;  // barrier: 0 gave up
};

// Every block of the (cooperative) launch arrives before any passes. False if the wait
// ran out; `target` counts this block's barriers in arrivals. A block that gave up arrives
// no more, so no other block gets past its next barrier: the phases behind a barrier only
// ever run on complete ones before it.
__device__ __forceinline__ bool grid_barrier(const LoopArgs& g, unsigned& target, LoopShared& sh, GraphCtl* ctl) {
  __syncthreads();
  if (threadIdx.x == 0) {
    target += gridDim.x;
    __threadfence();  // the block's writes (ordered before it by the barrier above)
    atomicAdd(g.bar, 1u);
    int polls = 0;
    unsigned v;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(g.bar) : "memory");
    } while ((int)(v - target) < 0 && ++polls < g.polls);
    sh.flag = polls < g.polls;
    if (polls >= g.polls) atomicMax(&ctl->abort, 3);
  }
  __syncthreads();
  return sh.flag != 0;
}

// Work lists of a rebuild pass (k_decide's, for at most 32 systems), by one warp.
__device__ __forceinline__ void loop_worklists(const DevArrays& a, const LoopArgs& g, const int* need) {
  const int lane = threadIdx.x & 31;
  const int k = lane < g.nsys ? a.sys_order[lane] : -1;
  const bool n = k >= 0 && need[k];
  const unsigned m = __ballot_sync(kFull, n);
  const int r = __popc(m & ((1u << lane) - 1u));
  int tiles = 0, chunks = 0;
  if (n) {
    const SysParams& P = a.params[k];
    tiles = P.ntiles;
    chunks = scan_chunks((int64_t)P.nc * P.nc * P.nc);
  }
  int ti = tiles, ci = chunks;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, ti, o), z = __shfl_up_sync(kFull, ci, o);
    if (lane >= o) { ti += y; ci += z; }
  }
  if (n) {
    g.rebuild_ids[r] = k;
    g.reb_pref[r] = ti - tiles;
    a.chunk_pref[r] = ci - chunks;
    g.reb_count[k] += 1;
    const_cast<int32_t*>(a.rebuild)[k] = 1;
    a.status[k] = SysStatus{0, 0, 0, 0};
  } else if (k >= 0) {
    const_cast<int32_t*>(a.rebuild)[k] = 0;
  }
  const int call = __shfl_sync(kFull, ci, 31);
  for (int q = lane; q < call * kChunkCopies; q += 32) a.chunk_sum[q] = 0;
  if (lane == 31) {
    const int nreb = __popc(m);
    g.reb_pref[nreb] = ti;
    a.chunk_pref[nreb] = ci;
    a.ctl->nreb = nreb;
    a.ctl->passes += 1;
  }
}

}  // namespace

template <bool kFP32, int T, bool kNvt>
__global__ void __launch_bounds__(kLoopBlock, T == 4 ? (kFP32 ? 4 : 3) : (kFP32 ? 3 : 2)) k_loop(DevArrays a, LoopArgs g) {
  extern __shared__ __align__(32) unsigned char smem[];
  __shared__ LoopShared sh;
  constexpr int CH = loop_chunk(T);
  float* ex_all = (float*)smem;
  WideShared& wide = *(WideShared*)smem;
  using Word = typename LoopWord<kFP32>::type;
  Word* lists = (Word*)(smem + loop_union_bytes(T));

  const int lane = threadIdx.x & 31, wv = threadIdx.x >> 5;
  const int sub = lane & (T - 1);                    // place among the particle's threads
  const int part = threadIdx.x / T;                  // particle of the block
  const int64_t slot = ((int64_t)blockIdx.x * kLoopBlock + threadIdx.x) / T;
  const int tile = (int)(slot / kTile);
  const int sys = tile < a.ntiles ? a.tile_sys[tile] : -1;  // uniform over the warp
  const SysParams& P = a.params[sys < 0 ? 0 : sys];
  const bool on = sys >= 0 && P.active;
  const int local = on ? (int)(slot - P.p_off) : 0;
  const bool act = on && local < P.n;
  const bool comp = act && sub < 3;  // this thread integrates axis `sub`
  const int64_t p_off = on ? P.p_off : 0;
  Word* list = lists + (size_t)part * g.stride;
  float* ex = ex_all + (size_t)part * loop_ex(T);
  const float qu = P.qunit, rc2f = P.rc2f, c2x8 = 8.0f * P.c2f;
  const long long rc2x = P.rc2fix;
  const FixC2 c2x{P.c2fix, P.c2fix_lo};
  const double dt = P.dt, h = P.hdt, qscale = P.qscale;

  int cur = g.cur;
  int niter = 0;                  // chunks of the warp's longest list
  double x = 0.0, v = 0.0, refd = 0.0;
  int q = 0, refq = 0;            // own shadow and its build-time value (FP32 form)
  long long ql = 0;               // own position in pair units (FP64 form)
  const int c = sub < 3 ? sub : 0;

  // The particle's state and list, after a rebuild or at the start. Lists are padded
  // with the particle itself to whole chunks.
  auto load_state = [&]() {
    int cnt = 0;
    if (act) {
      cnt = list_count(a, sys, slot, P.kmax);
      if (sub < 3) {
        x = ((const double*)&a.x[cur][slot])[c];
        v = ((const double*)&a.v[slot])[c];
        if (kFP32) {
          q = ((const int*)&a.xq[cur][slot])[c];
          refq = ((const int*)&a.xqref[slot])[c];
        } else {
          ql = ((const long long*)&a.xl[cur][slot])[c];
          refd = ((const double*)&a.xref[slot])[c];
        }
      }
    }
    const int most = __reduce_max_sync(kFull, cnt);
    niter = (most + CH * T - 1) / (CH * T);
    if (!check_ok(a, sys < 0 ? 0 : sys, niter * CH * T <= g.stride, kChkCount)) niter = g.stride / (CH * T);
    const uint32_t* lp = a.nbr + (on ? list_word(P.l_off, local / kTile, P.kmax, local % kTile, 0) : 0);
    for (int k = sub; k < niter * CH * T; k += T) {
      uint32_t e = (uint32_t)local;
      if (k < cnt) {
        e = lp[(int64_t)(k >> 2) * (4 * kTile) + (k & 3)];
        const uint32_t j = partner_slot(a, sys, e, P.n, (uint32_t)local);
        e = kFP32 ? j : (e & ~kIdxMask) | j;
      }
      list[k] = (Word)e;
    }
    __syncwarp();
  };

  // Force on the particle (axis c) at the positions of buffer cur.
  auto force = [&]() -> double {
    if constexpr (kFP32) {
      const int4* qs = a.xq[cur] + p_off;
      int4 qi;
      qi.x = __shfl_sync(kFull, q, 0, T);
      qi.y = __shfl_sync(kFull, q, 1, T);
      qi.z = __shfl_sync(kFull, q, 2, T);
      float f = 0.f;
      for (int it = 0; it < niter; ++it) {
        int4 qj[CH];
#pragma unroll
        for (int u = 0; u < CH; ++u) qj[u] = qs[list[(it * CH + u) * T + sub]];
#pragma unroll
        for (int u = 0; u < CH; ++u) {
          float4 d;
          d.w = pair_factor_fp32(qi, qj[u], qu, rc2f, c2x8, d.x, d.y, d.z);
          *(float4*)(ex + (u * T + sub) * 4) = d;
        }
        __syncwarp();
        if (sub < 3) {
#pragma unroll 8
          for (int m = 0; m < CH * T; ++m) f = fmaf(ex[4 * m + 3], ex[4 * m + c], f);
        }
        __syncwarp();
      }
      return f2d_bits(f);
    } else {
      const longlong4_32a* qs = a.xl[cur] + p_off;
      longlong4_32a qi;
      qi.x = __shfl_sync(kFull, ql, 0, T) - kFixBias;
      qi.y = __shfl_sync(kFull, ql, 1, T) - kFixBias;
      qi.z = __shfl_sync(kFull, ql, 2, T) - kFixBias;
      FixSum sx, sy, sz;
      int slow = 0, k0 = 0x7fffffff, k1 = 0x7fffffff;  // this thread's pairs for the FP64 pipe
#pragma unroll 1
      for (int it = 0; it < niter; ++it) {
        longlong4_32a qj[CH];
        uint32_t e[CH];
#pragma unroll
        for (int u = 0; u < CH; ++u) {
          e[u] = list[(it * CH + u) * T + sub];
          qj[u] = qs[e[u] & kIdxMask];
        }
#pragma unroll
        for (int u = 0; u < CH; ++u) {
          if (e[u] == (uint32_t)local) continue;  // padding
          if (fix_pair(qi, qj[u], e[u] >> kIdxBits, P.Lfix, rc2x, c2x, sx, sy, sz)) {
            if (slow == 0) k0 = (it * CH + u) * T + sub;
            else if (slow == 1) k1 = (it * CH + u) * T + sub;
            ++slow;
          }
        }
      }
#pragma unroll
      for (int o = T / 2; o > 0; o >>= 1) {
        sx.join(o);
        sy.join(o);
        sz.join(o);
      }
      double F = (c == 0 ? sx : c == 1 ? sy : sz).value24();
      if (__any_sync(kFull, slow > 0)) {
        // the FP64 pipe's pairs, in list order: the particle's threads take the lowest
        // entry left among them each time (a thread with more than two goes through
        // its whole list)
        const long long rc2b = __double_as_longlong(P.rc2);
        const double c8 = 8.0 * P.c2, L = P.L;
        double S0 = 0.0, S1 = 0.0, S2 = 0.0;
        const bool many = slow > 2;
        int next = many ? sub : k0;
        const int end = niter * CH * T;
        while (true) {
          if (many && next < end) {  // the next of this thread's entries that the fixed-point range leaves out
            for (; next < end; next += T) {
              const uint32_t e = list[next];
              if (e == (uint32_t)local) continue;
              FixSum t0, t1, t2;
              if (fix_pair(qi, qs[e & kIdxMask], e >> kIdxBits, P.Lfix, rc2x, c2x, t0, t1, t2)) break;
            }
          }
          int low = next < end ? next : 0x7fffffff;
#pragma unroll
          for (int o = T / 2; o > 0; o >>= 1) low = min(low, __shfl_xor_sync(kFull, low, o));
          if (!__any_sync(kFull, low != 0x7fffffff)) break;
          if (low != 0x7fffffff) {
            const uint32_t e = list[low];
            const double4_32a xi = a.x[cur][slot], xj = a.x[cur][p_off + (e & kIdxMask)];
            double dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
            const unsigned code = e >> kIdxBits;
            if (code) {
              dx = apply_image(dx, code & 3u, L);
              dy = apply_image(dy, (code >> 2) & 3u, L);
              dz = apply_image(dz, (code >> 4) & 3u, L);
            }
            const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
            if (__double_as_longlong(r2) < rc2b) {
              const double gg = force_factor<0>(r2, c8);
              S0 = fma(gg, dx, S0);
              S1 = fma(gg, dy, S1);
              S2 = fma(gg, dz, S2);
            }
            if (next == low) next = many ? next + T : (next == k0 ? k1 : 0x7fffffff);
          }
          __syncwarp();
        }
        const double S = c == 0 ? S0 : c == 1 ? S1 : S2;
        if (S0 != 0.0 || S1 != 0.0 || S2 != 0.0) F += S;
      }
      return F;
    }
  };

  for (int k = threadIdx.x; k < g.nsys; k += kLoopBlock) {
    sh.margin[k] = a.margin[k];
    sh.need[k] = (int)((g.rebuild0 >> k) & 1u);
  }
  const int target_steps = a.ctl->target;
  unsigned arrivals = 0;
  int done = 0, abort = 0;
  bool alive = true;
  // the decision's constants of system threadIdx.x
  bool dactive = false;
  double dthr = 0.0, ddt = 0.0;
  Thermo thermo{};  // system threadIdx.x's thermostat (every block keeps the same)
  if ((int)threadIdx.x < g.nsys) {
    const SysParams& Q = a.params[threadIdx.x];
    dactive = Q.active != 0;
    dthr = kFP32 ? Q.disp_thr : Q.skin;
    ddt = Q.dt;
    if (kNvt) thermo = g.thermo[threadIdx.x];
  }
  __syncthreads();

  // `halves` thermostat half steps at the current velocities; `turn` counts the calls.
  // False if the barrier gave up.
  int turn = 0;
  [[maybe_unused]] auto thermostat = [&](int halves) -> bool {
    if (blockIdx.x == 0)  // the next turn's sums: their last readers passed a barrier
      for (int m = threadIdx.x; m < kKeWords * g.nsys; m += kLoopBlock) g.ke[((turn + 1) % 3) * kKeWords * g.nsys + m] = 0ull;
    SquareSum s;
    if (comp) s.add(__dmul_rn(v, v));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s.join(o);
    if (lane == 0) {
      sh.ke[wv] = s;
      sh.sys[wv] = on ? sys : -1;
    }
    __syncthreads();
    if (wv == 0) {
      const int k = sh.sys[lane & (kLoopWarps - 1)];
      SquareSum m = sh.ke[lane & (kLoopWarps - 1)];
      unsigned long long* ke = g.ke + (turn % 3) * kKeWords * g.nsys;
      if (__all_sync(kFull, k == sh.sys[0])) {
#pragma unroll
        for (int o = kLoopWarps / 2; o > 0; o >>= 1) m.join(o);
        if (lane == 0 && k >= 0) add_limbs(ke + kKeWords * k, m);
      } else if (lane < kLoopWarps && k >= 0) {
        add_limbs(ke + kKeWords * k, m);
      }
    }
    if (!grid_barrier(g, arrivals, sh, a.ctl)) return false;
    if (dactive) {
      const unsigned long long* ke = g.ke + ((turn % 3) * g.nsys + threadIdx.x) * kKeWords;
      sh.scale[threadIdx.x] = thermo_halves(thermo, limbs_ke(ke), halves);
    }
    ++turn;
    __syncthreads();
    if (comp && sh.scale[sys] != 1.0) v *= sh.scale[sys];
    return true;
  };
  double fnow = 0.0;             // Nose-Hoover steps: the force at the current positions
  bool begun = false;            // the state is loaded
  bool pass = g.rebuild0 != 0u;  // a rebuild pass is due (the systems of sh.need)
  if (!pass) load_state();

  while (true) {
    if (pass) {
      const bool mine = on && sh.need[sys];
      if (begun && mine && comp) {
        ((double*)&a.x[cur][slot])[c] = x;
        ((double*)&a.v[slot])[c] = v;
      }
      if (blockIdx.x == 0 && wv == 0) loop_worklists(a, g, sh.need);
      if (!(alive = grid_barrier(g, arrivals, sh, a.ctl))) break;
      cell_count_pass<true>(a, cur);
      if (!(alive = grid_barrier(g, arrivals, sh, a.ctl))) break;
      cell_starts_pass(a, a.ctl->nreb, sh.ws);
      if (!(alive = grid_barrier(g, arrivals, sh, a.ctl))) break;
      scatter_pass<true>(a, cur);
      if (!(alive = grid_barrier(g, arrivals, sh, a.ctl))) break;
      cell_rank_pass<true>(a, cur);
      if (!(alive = grid_barrier(g, arrivals, sh, a.ctl))) break;
      build_lists_wide(a, cur, T == 32 ? 8 : T == 16 ? 16 : 32, wide);
      if (!(alive = grid_barrier(g, arrivals, sh, a.ctl))) break;
      if ((int)threadIdx.x < g.nsys && sh.need[threadIdx.x]) sh.margin[threadIdx.x] = a.margin[threadIdx.x];
      if (mine || !begun) load_state();
      abort = *(volatile int*)&a.ctl->abort;
      __syncthreads();
      if (abort) break;  // a list overflowed: the host grows it (uniform over the grid)
    }
    if constexpr (kNvt) {
      if (begun) {  // the step's closing half kick and the thermostat half steps
        if (on) {
          fnow = force();
          if (comp) v = fma(h, fnow, v);
        }
        if (!(alive = thermostat(done < target_steps ? 2 : g.halves_end))) break;
      } else {
        if (on) {
          if (!g.stored) fnow = force();
          else if (comp) fnow = ((const double*)&a.f[slot])[c];
        }
        if (g.open && !(alive = thermostat(1))) break;
      }
    }
    begun = true;
    if (done >= target_steps) break;
    unsigned long long d2 = 0ull;
    // block 0 clears the maximum of the next step: its last readers passed a barrier
    if (blockIdx.x == 0 && (int)threadIdx.x < g.nsys) g.disp[((done + 1) % 3) * g.nsys + threadIdx.x] = 0ull;
    if (on) {
      const bool first = done == 0;
      double F;
      if (kNvt) F = fnow;
      else if (first && g.stored) F = comp ? ((const double*)&a.f[slot])[c] : 0.0;
      else F = force();
      bool fine = true;
      long long s0 = 0;         // squared displacement of the axis (exact integer) ...
      double sd = 0.0;          // ... or its FP64 square, or the squared velocity
      if (comp) {
        if (!kNvt && (!first || g.steady)) v = fma(h, F, v);
        v = fma(h, F, v);
        const double xn = fma(dt, v, x);
        x = xn;
        fine = finite_bits(xn) && finite_bits(v);
        ((double*)&a.x[cur ^ 1][slot])[c] = xn;
        if (kFP32) {
          q = to_fixed(xn, qscale);
          ((int*)&a.xq[cur ^ 1][slot])[c] = q;
          const long long e = wrapped_diff(q, refq);
          s0 = e * e;
        } else {
          ql = to_fix(xn);
          ((long long*)&a.xl[cur ^ 1][slot])[c] = ql;
          if (!g.vmax) {
            const double e = __dsub_rn(xn, refd);
            sd = __dmul_rn(e, e);
          }
        }
        if (g.vmax) sd = __dmul_rn(v, v);
      }
      const unsigned bad = __ballot_sync(kFull, !fine);
      if (kFP32 && !g.vmax) {
        unsigned long long t = (unsigned long long)s0;
        t += (unsigned long long)__shfl_down_sync(kFull, s0, 1, T);
        t += (unsigned long long)__shfl_down_sync(kFull, s0, 2, T);
        d2 = t;  // valid at sub == 0
      } else {
        const double y = __shfl_down_sync(kFull, sd, 1, T), z = __shfl_down_sync(kFull, sd, 2, T);
        d2 = (unsigned long long)__double_as_longlong(__dadd_rn(__dadd_rn(sd, y), z));
      }
      if (sub != 0 || !act) d2 = 0ull;
      if (bad) {
        if (lane == 0) a.status[sys].nonfinite = 1;
        d2 = ~0ull;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(kFull, d2, o);
        d2 = y > d2 ? y : d2;
      }
    }
    // one atomic per block and system (on one word they complete one after the other)
    if (lane == 0) {
      sh.d2[wv] = d2;
      sh.sys[wv] = on ? sys : -1;
    }
    __syncthreads();
    if (wv == 0) {
      const int k = sh.sys[lane & (kLoopWarps - 1)];
      unsigned long long m = sh.d2[lane & (kLoopWarps - 1)];
      if (__all_sync(kFull, k == sh.sys[0])) {
#pragma unroll
        for (int o = kLoopWarps / 2; o > 0; o >>= 1) {
          const unsigned long long y = __shfl_xor_sync(kFull, m, o);
          m = y > m ? y : m;
        }
        if (lane == 0 && k >= 0 && m) atomicMax(&g.disp[(done % 3) * g.nsys + k], m);
      } else if (lane < kLoopWarps && k >= 0 && m) {
        atomicMax(&g.disp[(done % 3) * g.nsys + k], m);
      }
    }
    if (!grid_barrier(g, arrivals, sh, a.ctl)) { alive = false; break; }
    // the list-validity decision (k_decide's)
    bool need = false, stop = false;
    if ((int)threadIdx.x < g.nsys) {
      const int k = threadIdx.x;
      if (dactive) {
        const unsigned long long m2 = __ldcg(&g.disp[(done % 3) * g.nsys + k]);
        stop = m2 == ~0ull;
        if (g.vmax) {
          const double m = __dsub_rn(sh.margin[k], __dmul_rn(__dmul_rn(2.0, __dsqrt_rn(__longlong_as_double((long long)m2))), ddt));
          sh.margin[k] = m;
          need = !(m > 0.0);
        } else if (kFP32) {
          need = __ull2double_rn(m2) >= dthr;
        } else {
          need = !(2.0 * __dsqrt_rn(__longlong_as_double((long long)m2)) < dthr);
        }
      }
      sh.need[k] = need ? 1 : 0;
    }
    cur ^= 1;
    ++done;
    if (__syncthreads_or(stop)) { abort = 2; break; }
    pass = __syncthreads_or(need) != 0;
  }

  double F = 0.0;
  const bool close = !kNvt && alive && abort == 0 && g.finish;
  if (close && on) {
    F = force();
    if (comp) v = fma(h, F, v);
  }
  if (comp && (alive || begun)) {
    ((double*)&a.x[cur][slot])[c] = x;
    ((double*)&a.v[slot])[c] = v;
    if (!kFP32) ((int*)&a.xq[cur][slot])[c] = to_fixed(x, qscale);
    if (close || kNvt) ((double*)&a.f[slot])[c] = kNvt ? fnow : F;
  }
  if (blockIdx.x == 0) {
    if ((int)threadIdx.x < g.nsys) {
      a.margin[threadIdx.x] = sh.margin[threadIdx.x];
      if (kNvt) g.thermo[threadIdx.x] = thermo;
    }
    if (threadIdx.x == 0) {
      a.ctl->done = done;
      if (abort) atomicMax(&a.ctl->abort, abort);
    }
  }
}

// ---------------------------------------------------------------- launchers

namespace {
// At least one block: with no tiles its warps return at once (an empty arena).
inline unsigned tile_blocks(const DevArrays& a) {
  return (unsigned)std::max<int64_t>(1, ((int64_t)a.ntiles * kTile + kBlock - 1) / kBlock);
}
}  // namespace

// Positions as held (caller order, not wrapped) into the slots of a system whose
// list was just built, with their fixed-point shadows: a restored checkpoint.
__global__ void k_positions_by_id(DevArrays a, int cur, const double* __restrict__ x, int sys) {
  const SysParams P = a.params[sys];
  const int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (l >= P.n) return;
  const int64_t s = P.p_off + l;
  const int64_t i = a.id[s];
  const double4_32a xv = make_double4_32a(x[3 * i + 0], x[3 * i + 1], x[3 * i + 2], 0.0);
  a.x[cur][s] = xv;
  a.xq[cur][s] = fixed4(xv, P.qscale);
  if (a.xl[0]) a.xl[cur][s] = fix4(xv);
}

void launch_positions_by_id(const DevArrays& a, int cur, const double* x, int64_t sys_n, int sys, cudaStream_t s) {
  if (sys_n <= 0) return;
  k_positions_by_id<<<(unsigned)((sys_n + 255) / 256), 256, 0, s>>>(a, cur, x, sys);
}

void launch_from_caller(const DevArrays& a, int cur, const double* x, const double* v, int sys,
                        int64_t ntiles_sys, cudaStream_t s) {
  const int64_t n = ntiles_sys * kTile;
  k_from_caller<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, cur, x, v, sys);
}

void launch_state_to_caller(const DevArrays& a, int cur, double* x, double* v, int64_t sys_n, int sys, cudaStream_t s) {
  if (sys_n <= 0 || (!x && !v)) return;
  k_state_to_caller<<<(unsigned)((sys_n + 255) / 256), 256, 0, s>>>(a, cur, x, v, sys);
}

void launch_to_caller(const DevArrays& a, int cur, int which, double* out, int64_t sys_n, int sys,
                      int64_t, cudaStream_t s) {
  if (sys_n <= 0) return;
  k_to_caller<<<(unsigned)((sys_n + 255) / 256), 256, 0, s>>>(a, cur, which, out, sys);
}

// ------------------------------------------ graph-captured loop (decision)

// The list-validity decision after a drift (Sec. 2.1: the list is checked every
// step), for the graph-captured loop and for the host-driven one alike.
// Displacement rule: the FP32-force form compares the squared fixed-point
// displacement (an exact integer) with a threshold lowered by 4 units, the FP64
// forms test 2 sqrt(d2) >= skin. Velocity-bound rule (the DUTC check): the
// margin, the whole skin after a rebuild, shrinks by 2 v_max dt each step, and
// the list is rebuilt when it is no longer positive. Writes the rebuild flags
// and the rebuilding systems (in the order of sys_order: costliest list-build
// tiles first), resets the per-step maxima, and
// in a graph (reb_count set) counts steps, passes and rebuilds and sets the
// conditions of the rebuild node (h_if) and, after the second step of the loop
// body (last), of the loop node (h_loop). A non-finite position or velocity
// stops the loop (abort word 2).
__global__ void __launch_bounds__(1024) k_decide(DevArrays a, int nsys, int fp32, int vflag, int32_t* rebuild,
                                                 int32_t* rebuild_ids, int32_t* reb_pref, int32_t* reb_count,
                                                 cudaGraphConditionalHandle h_if,
                                                 cudaGraphConditionalHandle h_loop, int last) {
  GraphCtl* c = a.ctl;
  const bool graph = reb_count != nullptr;
  if (c->abort) {  // uniform over the block
    if (threadIdx.x == 0 && graph) {
      cudaGraphSetConditional(h_if, 0);
      if (last) cudaGraphSetConditional(h_loop, 0);
    }
    return;
  }
  __shared__ int wsum[32];
  __shared__ long long wsum64[32];
  __shared__ int base_s, bad_s, total_s;
  __shared__ long long total64_s;
  int32_t* chunk_pref = a.chunk_pref;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) { base_s = 0; bad_s = 0; }
  __syncthreads();
  for (int i0 = 0; i0 < nsys; i0 += (int)blockDim.x) {
    const int i = i0 + (int)threadIdx.x;
    const int k = i < nsys ? a.sys_order[i] : -1;
    int need = 0;
    if (k >= 0) {
      const unsigned long long d2 = a.disp2[k];
      a.disp2[k] = 0ull;
      const SysParams& P = a.params[k];
      if (P.active) {
        if (a.status[k].nonfinite) bad_s = 1;
        if (P.rule == 1) {
          // velocity bound (DUTC): the margin shrinks by 2 v_max dt per step; a
          // rebuild restores it (k_cell_starts)
          const double m =
              __dsub_rn(a.margin[k],
                        __dmul_rn(__dmul_rn(2.0, __dsqrt_rn(__longlong_as_double((long long)d2))), P.dt));
          a.margin[k] = m;
          need = (d2 == ~0ull || !(m > 0.0)) ? 1 : 0;
        } else if (fp32) {
          need = (d2 == ~0ull || __ull2double_rn(d2) >= P.disp_thr) ? 1 : 0;
        } else {
          need = !(2.0 * __dsqrt_rn(__longlong_as_double((long long)d2)) < P.skin) ? 1 : 0;
        }
      }
      rebuild[k] = need;
    }
    const unsigned b = __ballot_sync(kFull, need);
    if (lane == 0) wsum[w] = __popc(b);
    __syncthreads();
    if (w == 0) {
      const int v = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
      int incl = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
      }
      wsum[lane] = incl - v;
      if (lane == 31) total_s = incl;
    }
    __syncthreads();
    if (need) {
      rebuild_ids[base_s + wsum[w] + __popc(b & ((1u << lane) - 1u))] = k;
      if (graph) reb_count[k] += 1;
      a.status[k].overflow = 0;
      a.status[k].max_count = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) base_s += total_s;
    __syncthreads();
  }
  // prefixes of the rebuilding systems' tile counts (the rebuild kernels' work
  // list) and of their cell-chunk counts (the cell scan's work list), as one
  // scan of the pair packed in 64 bits
  const int nreb_all = base_s;
  long long carry = 0;
  for (int r0 = 0; r0 < nreb_all; r0 += (int)blockDim.x) {
    const int r = r0 + (int)threadIdx.x;
    long long v = 0;
    if (r < nreb_all) {
      const SysParams& P = a.params[rebuild_ids[r]];
      v = ((long long)scan_chunks((int64_t)P.nc * P.nc * P.nc) << 32) | (unsigned)P.ntiles;
    }
    long long incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) wsum64[w] = incl;
    __syncthreads();
    if (w == 0) {
      const long long ws = lane < (int)(blockDim.x >> 5) ? wsum64[lane] : 0;
      long long wi = ws;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, wi, o);
        if (lane >= o) wi += y;
      }
      wsum64[lane] = wi - ws;
      if (lane == 31) total64_s = wi;
    }
    __syncthreads();
    if (r < nreb_all) {
      const long long e = carry + wsum64[w] + incl - v;
      reb_pref[r] = (int32_t)(e & 0xffffffffll);
      chunk_pref[r] = (int32_t)(e >> 32);
    }
    carry += total64_s;
    __syncthreads();
  }
  // the pass's chunk totals start at zero (the count kernel adds to them)
  for (int q = (int)threadIdx.x; q < (int)(carry >> 32) * kChunkCopies; q += (int)blockDim.x) a.chunk_sum[q] = 0;
  if (threadIdx.x == 0) {
    const int nreb = base_s;
    reb_pref[nreb] = (int32_t)(carry & 0xffffffffll);
    chunk_pref[nreb] = (int32_t)(carry >> 32);
    *a.tile_next = 0;
    c->done += 1;
    if (bad_s) {
      c->abort = 2;
      if (graph) {
        cudaGraphSetConditional(h_if, 0);
        if (last) cudaGraphSetConditional(h_loop, 0);
      }
      return;
    }
    c->nreb = nreb;
    c->passes += nreb > 0 ? 1 : 0;
    c->flags = kStepKickA | kStepKickB | kStepDrift | vflag;
    if (graph) {
      cudaGraphSetConditional(h_if, nreb > 0 ? 1u : 0u);
      if (last) cudaGraphSetConditional(h_loop, c->done < c->target ? 1u : 0u);
    }
  }
}

void launch_decide(const DevArrays& a, int nsys, int fp32, int vflag, int32_t* rebuild, int32_t* rebuild_ids,
                   int32_t* reb_pref, int32_t* reb_count, cudaGraphConditionalHandle h_if,
                   cudaGraphConditionalHandle h_loop, int last, cudaStream_t s) {
  // one block; as many warps as the systems need (a single warp for one system)
  const int threads = std::max(32, std::min(1024, (nsys + 31) / 32 * 32));
  k_decide<<<1, threads, 0, s>>>(a, nsys, fp32, vflag, rebuild, rebuild_ids, reb_pref, reb_count, h_if, h_loop,
                                 last);
}

// Binning kernels of a rebuild pass: at most 64 blocks of 128 per SM; warps stride
// over the rebuilding systems' tiles.
inline unsigned bin_blocks(const DevArrays& a) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(((int64_t)a.ntiles + 3) / 4, 152 * 64));
}

void launch_cell_count(const DevArrays& a, int cur, cudaStream_t s) {
  k_cell_count<<<bin_blocks(a), kBlock, 0, s>>>(a, cur);
}
void launch_cell_scan(const DevArrays& a, int nreb, cudaStream_t s) {
  // blocks stride over the chunks: one wave of 8 blocks per SM at most
  const unsigned g = (unsigned)std::max(1, std::min(a.chunk_cap, 152 * 8));
  k_cell_starts<<<g, kScanBlock, 0, s>>>(a, nreb);
}
void launch_scatter(const DevArrays& a, int cur, cudaStream_t s) {
  k_scatter<<<bin_blocks(a), kBlock, 0, s>>>(a, cur);
}
void launch_cell_rank(const DevArrays& a, int cur, cudaStream_t s) {
  k_cell_rank<<<bin_blocks(a), kBlock, 0, s>>>(a, cur);
}
namespace {
inline unsigned blocks_of(const DevArrays& a, int block) {
  return (unsigned)std::max<int64_t>(1, ((int64_t)a.ntiles * kTile + block - 1) / block);
}
}  // namespace

// Rebuild passes: warps stride over (or fetch) the rebuilding systems' tiles, so
// the grids are sized to the GPU (two waves of resident warps) or to the arena's
// tiles if fewer.
constexpr int kSMs = 152;
inline unsigned reb_blocks(const DevArrays& a, int block, int blocks_per_sm) {
  const int64_t all = ((int64_t)a.ntiles * kTile + block - 1) / block;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(all, (int64_t)kSMs * blocks_per_sm * 2));
}

template <int VAR>
static void launch_build_list_v(const DevArrays& a, int cur, int block, cudaStream_t s) {
  switch (block) {
    case 64: k_build_list<64, VAR><<<reb_blocks(a, 64, 16), 64, 0, s>>>(a, cur); break;
    case 256: k_build_list<256, VAR><<<reb_blocks(a, 256, 4), 256, 0, s>>>(a, cur); break;
    default: k_build_list<128, VAR><<<reb_blocks(a, 128, 8), 128, 0, s>>>(a, cur); break;
  }
}

// The one-candidate-per-lane build takes the passes of arenas up to 1,300 tiles, where it
// is the faster one (rc 2.5, launch included): 22 against 74 us at 1000 particles, 24
// against 85 at 4000, 43 against 88 at 16,000, 74 against 95 at 32,000; from there a
// warp per tile fills the GPU (112 against 103 us at 64,000). Spans of 8 slots make
// enough blocks of small arenas; larger ones read the candidates of fewer runs (4000
// particles: 24 us at 8, 41 at 32; 32,000 particles: 94 at 8, 76 at 16, 74 at 32).
constexpr int kWideMaxTiles = 1300;
inline int wide_span(int ntiles) { return ntiles <= 152 ? 8 : ntiles <= 304 ? 16 : 32; }

void launch_build_list(const DevArrays& a, int cur, const Tuning& tu, cudaStream_t s) {
  switch (tu.list_variant) {
    case 5:
      if (a.ntiles <= kWideMaxTiles) {
        const int span = wide_span(a.ntiles);
        k_build_list_wide<<<(unsigned)std::max(1, std::min(a.ntiles * (kTile / span), kSMs * 8)), kWideBlock, 0, s>>>(
            a, cur, span);
        break;
      }
      switch (tu.list_block) {
        case 64: k_build_list_staged<64><<<reb_blocks(a, 64, 16), 64, 0, s>>>(a, cur); break;
        case 256: k_build_list_staged<256><<<reb_blocks(a, 256, 4), 256, 0, s>>>(a, cur); break;
        default: k_build_list_staged<128><<<reb_blocks(a, 128, 8), 128, 0, s>>>(a, cur); break;
      }
      break;
    case 4:
      switch (tu.list_block) {
        case 64: k_build_list_warp<64><<<reb_blocks(a, 64, 16), 64, 0, s>>>(a, cur); break;
        case 256: k_build_list_warp<256><<<reb_blocks(a, 256, 4), 256, 0, s>>>(a, cur); break;
        default: k_build_list_warp<128><<<reb_blocks(a, 128, 8), 128, 0, s>>>(a, cur); break;
      }
      break;
    case 1: launch_build_list_v<1>(a, cur, tu.list_block, s); break;
    case 2: launch_build_list_v<2>(a, cur, tu.list_block, s); break;
    case 3: launch_build_list_v<3>(a, cur, tu.list_block, s); break;
    default: launch_build_list_v<0>(a, cur, tu.list_block, s); break;
  }
}
template <int MODE, bool QUEUE, bool FIXED = false>
static void launch_step_fp64_m(const DevArrays& a, int cur, double ka, double kb, int flags, int block,
                               cudaStream_t s) {
  switch (block) {
    case 64: k_step_fp64<64, MODE, QUEUE, FIXED><<<blocks_of(a, 64), 64, 0, s>>>(a, cur, ka, kb, flags); break;
    case 256: k_step_fp64<256, MODE, QUEUE, FIXED><<<blocks_of(a, 256), 256, 0, s>>>(a, cur, ka, kb, flags); break;
    default: k_step_fp64<128, MODE, QUEUE, FIXED><<<blocks_of(a, 128), 128, 0, s>>>(a, cur, ka, kb, flags); break;
  }
}

template <bool QUEUE>
static void launch_step_fp64_q(const DevArrays& a, int cur, double ka, double kb, int flags, const Tuning& tu,
                               int mode, cudaStream_t s) {
  switch (mode) {
    case 1: launch_step_fp64_m<1, QUEUE>(a, cur, ka, kb, flags, tu.step_block, s); break;
    case 2: launch_step_fp64_m<2, QUEUE>(a, cur, ka, kb, flags, tu.step_block, s); break;
    case 3: launch_step_fp64_m<3, QUEUE>(a, cur, ka, kb, flags, tu.step_block, s); break;
    case 4: launch_step_fp64_m<4, QUEUE>(a, cur, ka, kb, flags, tu.step_block, s); break;
    default:
      if (a.xl[0]) launch_step_fp64_m<0, QUEUE, true>(a, cur, ka, kb, flags, tu.step_block, s);
      else launch_step_fp64_m<0, QUEUE>(a, cur, ka, kb, flags, tu.step_block, s);
      break;
  }
}

void launch_step_fp64(const DevArrays& a, int cur, double ka, double kb, int flags, const Tuning& tu,
                      int mode, cudaStream_t s) {
  if (tu.fp64_queue) launch_step_fp64_q<true>(a, cur, ka, kb, flags, tu, mode, s);
  else launch_step_fp64_q<false>(a, cur, ka, kb, flags, tu, mode, s);
}
template <int MODE>
static void launch_force_half_fp64_m(const DevArrays& a, int cur, int flags, int block, cudaStream_t s) {
  switch (block) {
    case 64: k_force_half_fp64<64, MODE><<<blocks_of(a, 64), 64, 0, s>>>(a, cur, flags); break;
    case 256: k_force_half_fp64<256, MODE><<<blocks_of(a, 256), 256, 0, s>>>(a, cur, flags); break;
    default: k_force_half_fp64<128, MODE><<<blocks_of(a, 128), 128, 0, s>>>(a, cur, flags); break;
  }
}

void launch_step_half(const DevArrays& a, int cur, int flags, const Tuning& tu, int precision, cudaStream_t s) {
  if (precision == 1) {
    switch (tu.step_block) {
      case 64: k_force_half_fp32<64><<<blocks_of(a, 64), 64, 0, s>>>(a, cur, flags); break;
      case 256: k_force_half_fp32<256><<<blocks_of(a, 256), 256, 0, s>>>(a, cur, flags); break;
      default: k_force_half_fp32<128><<<blocks_of(a, 128), 128, 0, s>>>(a, cur, flags); break;
    }
    k_integrate_half<true><<<tile_blocks(a), kBlock, 0, s>>>(a, cur, flags);
    return;
  }
  switch (precision) {
    case 2: launch_force_half_fp64_m<1>(a, cur, flags, tu.step_block, s); break;
    case 3: launch_force_half_fp64_m<2>(a, cur, flags, tu.step_block, s); break;
    case 4: launch_force_half_fp64_m<3>(a, cur, flags, tu.step_block, s); break;
    case 5: launch_force_half_fp64_m<4>(a, cur, flags, tu.step_block, s); break;
    default: launch_force_half_fp64_m<0>(a, cur, flags, tu.step_block, s); break;
  }
  k_integrate_half<false><<<tile_blocks(a), kBlock, 0, s>>>(a, cur, flags);
}

void launch_step_fp32(const DevArrays& a, int cur, double ka, double kb, int flags, const Tuning& tu,
                      cudaStream_t s) {
  const int b = tu.step_block, g = tu.step_groups;
#define LJMD_STEP32(B, G, H) k_step_fp32<B, G, H><<<blocks_of(a, B), B, 0, s>>>(a, cur, ka, kb, flags)
#define LJMD_STEP32B(G, H)             \
  if (b == 64) LJMD_STEP32(64, G, H);  \
  else if (b == 256) LJMD_STEP32(256, G, H); \
  else LJMD_STEP32(128, G, H)
  if (tu.step_hint) {
    if (g == 2) { LJMD_STEP32B(2, true); } else { LJMD_STEP32B(1, true); }
  } else {
    if (g == 2) { LJMD_STEP32B(2, false); } else { LJMD_STEP32B(1, false); }
  }
#undef LJMD_STEP32B
#undef LJMD_STEP32
}
namespace {
template <bool kFP32, int T, bool kNvt>
cudaError_t loop_setup_k(size_t bytes, int* blocks_per_sm) {
  // The limit belongs to the kernel, not to a launch: always the largest one, so that
  // threads with other sizes do not lower it under each other's launches.
  int dev = 0, optin = 0;
  cudaFuncAttributes fa{};
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_loop<kFP32, T, kNvt>);
  if (e != cudaSuccess) return e;
  const int most = optin - (int)fa.sharedSizeBytes;
  if (bytes > (size_t)most) return cudaErrorInvalidValue;
  e = cudaFuncSetAttribute(k_loop<kFP32, T, kNvt>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_loop<kFP32, T, kNvt>, kLoopBlock, bytes);
  return e;
}
template <bool kFP32, int T>
cudaError_t loop_setup(int kmax, int* stride, size_t* bytes, int* blocks_per_sm) {
  const int unit = loop_chunk(T) * T;
  int st = (kmax + unit - 1) / unit * unit;  // whole chunks, the particles of a warp on different banks
  st += (T - st % 32 + 32) % 32;
  *stride = st;
  *bytes = loop_union_bytes(T) + sizeof(typename LoopWord<kFP32>::type) * (size_t)st * (kLoopBlock / T);
  // both kinds of steps take the plan
  int plain = 0, nvt = 0;
  cudaError_t e = loop_setup_k<kFP32, T, false>(*bytes, &plain);
  if (e == cudaSuccess) e = loop_setup_k<kFP32, T, true>(*bytes, &nvt);
  *blocks_per_sm = std::min(plain, nvt);
  return e;
}
template <bool kFP32>
cudaError_t loop_setup(int T, int kmax, int* stride, size_t* bytes, int* bps) {
  switch (T) {
    case 32: return loop_setup<kFP32, 32>(kmax, stride, bytes, bps);
    case 16: return loop_setup<kFP32, 16>(kmax, stride, bytes, bps);
    case 8: return loop_setup<kFP32, 8>(kmax, stride, bytes, bps);
    default: return loop_setup<kFP32, 4>(kmax, stride, bytes, bps);
  }
}
template <bool kFP32, bool kNvt>
const void* loop_kernel(int T) {
  return T == 32 ? (const void*)k_loop<kFP32, 32, kNvt> : T == 16 ? (const void*)k_loop<kFP32, 16, kNvt>
         : T == 8 ? (const void*)k_loop<kFP32, 8, kNvt> : (const void*)k_loop<kFP32, 4, kNvt>;
}
unsigned loop_blocks(int ntiles, int T) { return (unsigned)(((int64_t)ntiles * kTile * T + kLoopBlock - 1) / kLoopBlock); }
}  // namespace

// A launch takes the most threads per particle whose blocks are all resident at once: alone
// on the device 32 and 16 up to two blocks per SM (2,432 and 4,864 particles), 8 and 4 up
// to what fits (three or four blocks of the FP32 form, 38,912 particles; three of the FP64
// form, 29,184).
void loop_plans(int fp32, int ntiles, int kmax, LoopPlan* plans) {
  int dev = 0, sms = 0;
  const bool fits = ntiles > 0 && (int64_t)ntiles * kTile <= 65535 /* LoopWord */ && cudaGetDevice(&dev) == cudaSuccess &&
                    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
  for (int m = 0; m < kLoopPlans; ++m) {
    const int T = 32 >> m;
    LoopPlan& p = plans[m];
    p = LoopPlan{T, 0, 0, 0, 0};
    if (!fits) continue;
    size_t bytes = 0;
    int bps = 0;
    const cudaError_t e = fp32 ? loop_setup<true>(T, kmax, &p.stride, &bytes, &bps) : loop_setup<false>(T, kmax, &p.stride, &bytes, &bps);
    if (e != cudaSuccess) continue;
    p.blocks = (int)loop_blocks(ntiles, T);
    p.resident = sms * bps;
    p.alone = T >= 16 ? sms * std::min(bps, 2) : p.resident;
  }
  cudaGetLastError();
}

cudaError_t launch_loop(const DevArrays& a, const LoopArgs& g, cudaStream_t s) {
  DevArrays ac = a;
  LoopArgs gc = g;
  void* args[] = {&ac, &gc};
  const void* fn = g.thermo ? (g.fp32 ? loop_kernel<true, true>(g.lanes) : loop_kernel<false, true>(g.lanes))
                            : (g.fp32 ? loop_kernel<true, false>(g.lanes) : loop_kernel<false, false>(g.lanes));
  const size_t word = g.fp32 ? sizeof(LoopWord<true>::type) : sizeof(LoopWord<false>::type);
  const size_t bytes = loop_union_bytes(g.lanes) + word * (size_t)g.stride * (kLoopBlock / g.lanes);
  return cudaLaunchCooperativeKernel(fn, dim3(loop_blocks(a.ntiles, g.lanes)), dim3(kLoopBlock), args, bytes, s);
}

void launch_pe_virial(const DevArrays& a, int cur, int with_pairs, const int32_t* select, cudaStream_t s) {
  const longlong4_32a* xl = a.xl[0] ? a.xl[cur] : reinterpret_cast<const longlong4_32a*>(a.vtmp);
  if (with_pairs && !a.xl[0]) k_fix_positions<<<tile_blocks(a), kBlock, 0, s>>>(a, cur, select);
  k_pe_virial<<<tile_blocks(a), kBlock, 0, s>>>(a, cur, with_pairs, select, xl);
}

// v *= factor for every particle of the systems with scale[sys] != 1.
__global__ void k_scale_v(DevArrays a, const double* __restrict__ scale) {
  TileCtx t;
  SysParams P;
  if (!tile_ctx(a, t, P) || !t.act) return;
  const double f = scale[t.sys];
  if (f == 1.0) return;
  double4_32a v = a.v[t.s];
  v.x *= f;
  v.y *= f;
  v.z *= f;
  a.v[t.s] = v;
}

void launch_scale_v(const DevArrays& a, const double* scale, cudaStream_t s) {
  k_scale_v<<<tile_blocks(a), kBlock, 0, s>>>(a, scale);
}
void launch_thermostat(const DevArrays& a, int nsys, Thermo* thermo, int halves, unsigned long long* ke, double* scale,
                       cudaStream_t s) {
  // at most four blocks per SM, so that few warps meet on a system's sums
  const unsigned g = (unsigned)std::max(1, std::min((a.ntiles + 7) / 8, kSMs * 4));
  k_ke_limbs<<<g, 256, 0, s>>>(a, ke);
  k_thermostat<<<(unsigned)((nsys + 127) / 128), 128, 0, s>>>(a, nsys, thermo, halves, ke, scale);
  launch_scale_v(a, scale, s);
}

void launch_pair_stats(const DevArrays& a, int cur, unsigned long long* out2, cudaStream_t s) {
  k_pair_stats<<<tile_blocks(a), kBlock, 0, s>>>(a, cur, out2);
}
void launch_reduce_obs(const DevArrays& a, const int32_t* work, int nsel, int nchunks, double* chunk3, double* out3,
                       cudaStream_t s) {
  if (nsel <= 0 || nchunks <= 0) return;
  k_obs_chunks<<<nchunks, kObsChunk, 0, s>>>(a, work, nsel, chunk3);
  k_obs_final<<<nsel, 256, 0, s>>>(work, nsel, chunk3, out3);
}

}  // namespace ljmd
