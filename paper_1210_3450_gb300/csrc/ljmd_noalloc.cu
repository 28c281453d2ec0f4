// Allocation-free force entry point (md_forces_noalloc).
//
// Some callers cannot let a library call cudaMalloc: applications whose device
// memory is owned by their own allocator or memory pool (which must account for
// every byte and may already hold nearly all of it), and code that cannot afford
// the implicit device-wide synchronisation of cudaMalloc / cudaFree. For them this
// file offers one call that computes truncated-LJ forces for positions the caller
// passes in, into a force array the caller passes in, and keeps every piece of
// working memory in one fixed file-scope device array instead of allocating it.
//
// The working memory (cell counters, cell starts, per-particle cells, the
// scattered caller indices, the cell-sorted copy of the positions) lives in
// g_noalloc_scratch below; every GPU
// that loads this library holds that array until the process exits. Host code
// cannot use the symbol g_noalloc_scratch as a device address (it names a host
// stand-in), so the device address is looked up with cudaGetSymbolAddress, once
// per device, with that device current, on the first call made on that device.
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>
#include <string>

#include "ljmd.h"
#include "ljmd_dev.cuh"
#include "ljmd_engine.h"
#include "ljmd_fixed.cuh"
#include "ljmd_math.cuh"

namespace ljmd {
namespace {

constexpr int64_t kNaMaxN = 65536;      // particles per call
constexpr int64_t kNaMaxCells = 32768;  // cell grid of at most 32^3 cells
constexpr int kNaMaxDevices = 64;

// Layout of the scratch array (bytes, each part 256-aligned).
constexpr size_t kOffCount = 0;                                          // int[kNaMaxCells]
constexpr size_t kOffStart = kOffCount + 4 * kNaMaxCells;                // int[kNaMaxCells + 1]
constexpr size_t kOffCell = kOffStart + 4 * (kNaMaxCells + 256);         // int[kNaMaxN]
constexpr size_t kOffIdx = kOffCell + 4 * kNaMaxN;                       // int[kNaMaxN]
constexpr size_t kOffPos = kOffIdx + 4 * kNaMaxN;                        // double4_32a[kNaMaxN]
constexpr size_t kScratchBytes = kOffPos + 32 * kNaMaxN;                 // 3.0 MiB

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

struct NaParams {
  double L, inv_cs, rc2, c2x8;
  int n, nc;
  // fixed-point form (k_na_force_fixed)
  long long Lfix, rc2fix;
  FixC2 c2fix;
  float rc2q;  // (rc + 2^-24)^2 (1 + 1e-5) in units of 2^-56
};

struct NaScratch {
  int* count;
  int* start;
  int* cell;
  int* idx;          // caller indices scattered into cell order (arbitrary within a cell)
  double4_32a* pos;  // wrapped positions in cell order, by caller index within a cell; w = caller index
                     // (the fixed-point form keeps them there in pair units, as longlong4_32a)
};

__device__ __forceinline__ NaScratch na_view(unsigned char* base) {
  NaScratch s;
  s.count = (int*)(base + kOffCount);
  s.start = (int*)(base + kOffStart);
  s.cell = (int*)(base + kOffCell);
  s.idx = (int*)(base + kOffIdx);
  s.pos = (double4_32a*)(base + kOffPos);
  return s;
}

__global__ void k_na_clear(unsigned char* base, int ncell) {
  NaScratch s = na_view(base);
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ((ncell + 3) & ~3); c += gridDim.x * blockDim.x) s.count[c] = 0;
}

__global__ void k_na_bin(unsigned char* base, NaParams p, const double* __restrict__ x) {
  NaScratch s = na_view(base);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= p.n) return;
  const double4_32a w = make_double4_32a(wrap_fast(x[3 * i + 0], p.L), wrap_fast(x[3 * i + 1], p.L),
                                         wrap_fast(x[3 * i + 2], p.L), 0.0);
  const int c = p.nc > 1 ? cell_of(w, p.inv_cs, p.nc) : 0;
  s.cell[i] = c;
  atomicAdd(&s.count[c], 1);
}

// Single block, four cells per thread: exclusive scan of the counts; counts become fill
// counters.
__global__ void __launch_bounds__(1024) k_na_scan(unsigned char* base, int ncell) {
  NaScratch s = na_view(base);
  __shared__ int wsum[32];
  __shared__ int total;
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  int carry = 0;
  for (int b0 = 0; b0 < ncell; b0 += 4096) {
    const int c = b0 + 4 * tid;
    int4 v = make_int4(0, 0, 0, 0);
    if (c < ncell) v = *reinterpret_cast<const int4*>(s.count + c);  // (the clear covers whole fours)
    const int sum = v.x + v.y + v.z + v.w;
    int incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[wp] = incl;
    __syncthreads();
    if (wp == 0) {
      const int ws = wsum[lane];
      int wi = ws;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, wi, o);
        if (lane >= o) wi += y;
      }
      wsum[lane] = wi - ws;
      if (lane == 31) total = wi;
    }
    __syncthreads();
    if (c < ncell) {
      const int e = carry + wsum[wp] + incl - sum;
      *reinterpret_cast<int4*>(s.start + c) = make_int4(e, e + v.x, e + v.x + v.y, e + v.x + v.y + v.z);
      *reinterpret_cast<int4*>(s.count + c) = make_int4(0, 0, 0, 0);
    }
    carry += total;
    __syncthreads();
  }
  if (tid == 0) s.start[ncell] = carry;  // after the fours, whose last entries may lie past ncell
}

// Caller indices into their cells' ranges, in arrival order.
__global__ void k_na_scatter(unsigned char* base, NaParams p) {
  NaScratch s = na_view(base);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= p.n) return;
  const int c = s.cell[i];
  s.idx[s.start[c] + atomicAdd(&s.count[c], 1)] = i;
}

// Each particle's place in its cell is the number of the cell's particles with a
// smaller caller index, so the cell-sorted positions, and with them the order of
// every force sum, do not depend on the order of the atomics above: the same
// positions give the same forces bit for bit.
template <bool kFixed>
__global__ void k_na_rank(unsigned char* base, NaParams p, const double* __restrict__ x) {
  NaScratch s = na_view(base);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= p.n) return;
  const int c = s.cell[i];
  const int lo = s.start[c], hi = s.start[c + 1];
  int rank = 0;
  for (int q = lo; q < hi; ++q) rank += s.idx[q] < i ? 1 : 0;
  const double wx = wrap_fast(x[3 * i + 0], p.L), wy = wrap_fast(x[3 * i + 1], p.L), wz = wrap_fast(x[3 * i + 2], p.L);
  // (a position that is not finite has no pairs: its index is stored inverted)
  if (kFixed)
    reinterpret_cast<longlong4_32a*>(s.pos)[lo + rank] =
        longlong4_32a{to_fix(wx), to_fix(wy), to_fix(wz), finite_bits(wx) && finite_bits(wy) && finite_bits(wz) ? i : ~i};
  else s.pos[lo + rank] = make_double4_32a(wx, wy, wz, (double)i);
}

// Force on caller particle i from every j in the 27 neighbour cells (or from all
// particles when nc == 1), minimum image, r < rc: the same pair force as the
// list-based kernels, F_i = sum_j (24 r^-8 - 48 r^-14 + 8 c2)(x_j - x_i).
__global__ void k_na_force(unsigned char* base, NaParams p, const double* __restrict__ x,
                           double* __restrict__ f) {
  NaScratch s = na_view(base);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= p.n) return;
  const double xi = wrap_full(x[3 * i + 0], p.L), yi = wrap_full(x[3 * i + 1], p.L),
               zi = wrap_full(x[3 * i + 2], p.L);
  const long long rc2b = __double_as_longlong(p.rc2);
  double fx = 0.0, fy = 0.0, fz = 0.0;
  auto pair = [&](const double4_32a& q, double sx, double sy, double sz) {
    if ((int)q.w == i) return;
    const double dx = (q.x - xi) + sx, dy = (q.y - yi) + sy, dz = (q.z - zi) + sz;
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    if (__double_as_longlong(r2) < rc2b) {
      const double ir2 = rcp_f64(r2);
      const double ir4 = ir2 * ir2;
      const double g = fma(ir4 * ir4, fma(-48.0, ir4 * ir2, 24.0), p.c2x8);
      fx = fma(g, dx, fx);
      fy = fma(g, dy, fy);
      fz = fma(g, dz, fz);
    }
  };
  if (p.nc > 1) {
    const int nc = p.nc;
    const int ci = s.cell[i];
    const int cx = ci % nc, cy = (ci / nc) % nc, cz = ci / (nc * nc);
    for (int oz = -1; oz <= 1; ++oz) {
      int nz = cz + oz;
      double sz = 0.0;
      if (nz < 0) { nz += nc; sz = -p.L; } else if (nz >= nc) { nz -= nc; sz = p.L; }
      for (int oy = -1; oy <= 1; ++oy) {
        int ny = cy + oy;
        double sy = 0.0;
        if (ny < 0) { ny += nc; sy = -p.L; } else if (ny >= nc) { ny -= nc; sy = p.L; }
        for (int ox = -1; ox <= 1; ++ox) {
          int nx = cx + ox;
          double sx = 0.0;
          if (nx < 0) { nx += nc; sx = -p.L; } else if (nx >= nc) { nx -= nc; sx = p.L; }
          const int c = nx + nc * (ny + nc * nz);
          for (int q = s.start[c]; q < s.start[c + 1]; ++q) pair(s.pos[q], sx, sy, sz);
        }
      }
    }
  } else {
    for (int q = 0; q < p.n; ++q) {
      const double4_32a pj = s.pos[q];
      pair(pj, -p.L * rint((pj.x - xi) / p.L), -p.L * rint((pj.y - yi) / p.L),
           -p.L * rint((pj.z - zi) / p.L));
    }
  }
  f[3 * i + 0] = fx;
  f[3 * i + 1] = fy;
  f[3 * i + 2] = fz;
}

// The same forces in the fixed-point arithmetic of ljmd_fixed.cuh, T threads per particle.
// One thread per particle in caller order tested all 355 candidates of the 27 cells in
// FP64 and ran the force body for whichever lane was inside: 1,150 us at 65,536
// particles, 600 us at 500 (two blocks of threads). Here the particles are taken in cell
// order, the candidates of a row of cells are tested on the high words of their
// positions (unit 2^-28) in float against rc^2 and a margin, and each thread queues its
// maybe-inside ones and works them off behind the tests. The sums are exact integers,
// the pairs closer than the fixed-point range are added in a fixed order.
constexpr int kNaBlock = 128;
constexpr int kNaQueue = 32;
// Candidates that a thread loads at a time (one at a time waits for L2: 140 us a call at
// 65,536 particles, 4 threads each; two 116, three 109, four 104. With more threads a row
// gives each fewer: 4,000 particles, 8 threads each, 50.8 us, three 41.1, four 42.6;
// 500 particles, 32 threads each, 36.4, 34.8, 36.9; with a factor of two parts, with the
// present one 3 % more).
__host__ __device__ constexpr int na_loads(int T) { return T <= 4 ? 4 : 3; }

template <int T>
__global__ void __launch_bounds__(kNaBlock) k_na_force_fixed(unsigned char* base, NaParams p,
                                                             const double* __restrict__ x, double* __restrict__ f) {
  constexpr int K = na_loads(T);
  __shared__ uint32_t queue[kNaQueue][kNaBlock];
  NaScratch s = na_view(base);
  const longlong4_32a* pos = reinterpret_cast<const longlong4_32a*>(s.pos);
  const int t = (blockIdx.x * kNaBlock + threadIdx.x) / T, sub = threadIdx.x & (T - 1);
  const bool act = t < p.n;
  uint32_t* qme = &queue[0][threadIdx.x];
  FixSum sx, sy, sz;
  double Fx = 0.0, Fy = 0.0, Fz = 0.0;
  int inside = 0, i = 0;
  longlong4_32a qi{0, 0, 0, 0};
  auto fp64_pair = [&](uint32_t j, unsigned code) {
    const int64_t k = pos[j].w;
    const double dx = apply_image(wrap_full(x[3 * k + 0], p.L) - wrap_full(x[3 * (int64_t)i + 0], p.L), code & 3u, p.L);
    const double dy = apply_image(wrap_full(x[3 * k + 1], p.L) - wrap_full(x[3 * (int64_t)i + 1], p.L), (code >> 2) & 3u, p.L);
    const double dz = apply_image(wrap_full(x[3 * k + 2], p.L) - wrap_full(x[3 * (int64_t)i + 2], p.L), (code >> 4) & 3u, p.L);
    const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
    if (__double_as_longlong(r2) < __double_as_longlong(p.rc2)) {
      const double ir2 = rcp_f64(r2);
      const double ir4 = ir2 * ir2;
      const double g = fma(ir4 * ir4, fma(-48.0, ir4 * ir2, 24.0), p.c2x8);
      Fx = fma(g, dx, Fx);
      Fy = fma(g, dy, Fy);
      Fz = fma(g, dz, Fz);
    }
  };
  // All pairs of the particle; fixed: in fixed point where the range allows it.
  auto sum = [&](bool fixed) {
    int qn = 0;
    auto drain = [&]() {
      for (int k = 0; k < qn; ++k) {
        const uint32_t e = qme[k * kNaBlock];
        const uint32_t j = e & kIdxMask;
        if (pos[j].w < 0) continue;
        if (!fixed || fix_pair(qi, pos[j], e >> kIdxBits, p.Lfix, p.rc2fix, p.c2fix, sx, sy, sz)) fp64_pair(j, e >> kIdxBits);
      }
      inside += qn;
      qn = 0;
    };
    const int nc = p.nc;
    const int ci = s.cell[i];
    const int cx = ci % nc, cy = (ci / nc) % nc, cz = ci / (nc * nc);
    const int hx = (int)((qi.x + kFixBias) >> 32), hy = (int)((qi.y + kFixBias) >> 32), hz = (int)((qi.z + kFixBias) >> 32);
    const int hL = (int)(p.Lfix >> 32);
    for (int r = 0; r < 9; ++r) {
      int nz = cz + r / 3 - 1, ny = cy + r % 3 - 1;
      unsigned row = 0u;  // image code: 1 adds L, 2 subtracts it
      if (nz < 0) { nz += nc; row |= 32u; } else if (nz >= nc) { nz -= nc; row |= 16u; }
      if (ny < 0) { ny += nc; row |= 8u; } else if (ny >= nc) { ny -= nc; row |= 4u; }
      const int* st = s.start + nc * (ny + nc * nz);
      for (int part = 0; part < 2; ++part) {  // a row that wraps in x has two pieces
        int c0 = cx - 1, c1 = cx + 2;
        unsigned code = row;
        if (cx == 0) {
          if (part == 0) { c0 = nc - 1; c1 = nc; code |= 2u; }
          else { c0 = 0; c1 = 2; }
        } else if (cx == nc - 1) {
          if (part == 0) { c0 = nc - 2; c1 = nc; }
          else { c0 = 0; c1 = 1; code |= 1u; }
        } else if (part == 1) {
          break;
        }
        // the particle's high words, shifted against the image
        const int px = (code & 3u) == 1u ? hx - hL : ((code & 3u) == 2u ? hx + hL : hx);
        const int py = (code & 12u) == 4u ? hy - hL : ((code & 12u) == 8u ? hy + hL : hy);
        const int pz = (code & 48u) == 16u ? hz - hL : ((code & 48u) == 32u ? hz + hL : hz);
        const int hi = st[c1];
        for (int j = st[c0] + sub; j < hi; j += K * T) {
          if (qn > kNaQueue - K) drain();
          int c[K][3];  // high words (the first candidate's again past the row's end)
#pragma unroll
          for (int u = 0; u < K; ++u) {
            const int ju = j + u * T < hi ? j + u * T : j;
            const int* w = reinterpret_cast<const int*>(pos + ju);  // little-endian halves
            c[u][0] = w[1]; c[u][1] = w[3]; c[u][2] = w[5];
          }
#pragma unroll
          for (int u = 0; u < K; ++u) {
            const int ju = j + u * T;
            const float ax = (float)wrapped_diff(c[u][0], px), ay = (float)wrapped_diff(c[u][1], py),
                        az = (float)wrapped_diff(c[u][2], pz);
            if (fmaf(az, az, fmaf(ay, ay, ax * ax)) < p.rc2q && ju != t && (u == 0 || ju < hi)) {
              qme[qn * kNaBlock] = (uint32_t)ju | (code << kIdxBits);
              ++qn;
            }
          }
        }
      }
    }
    drain();
  };
  if (act) {
    qi = pos[t];
    i = (int)(qi.w < 0 ? ~qi.w : qi.w);
    qi.x -= kFixBias;
    qi.y -= kFixBias;
    qi.z -= kFixBias;
    if (qi.w >= 0) sum(true);
  }
  int all = inside;
#pragma unroll
  for (int o = T / 2; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
  if (act && all > kFixMaxList) {  // more pairs than the 96-bit sums take
    Fx = Fy = Fz = 0.0;
    sum(false);
  }
#pragma unroll
  for (int o = T / 2; o > 0; o >>= 1) {
    sx.join(o);
    sy.join(o);
    sz.join(o);
    Fx += __shfl_xor_sync(0xffffffffu, Fx, o);
    Fy += __shfl_xor_sync(0xffffffffu, Fy, o);
    Fz += __shfl_xor_sync(0xffffffffu, Fz, o);
  }
  if (act && sub == 0) {
    if (all <= kFixMaxList) {
      const bool some = Fx != 0.0 || Fy != 0.0 || Fz != 0.0;
      const double gx = sx.value24(), gy = sy.value24(), gz = sz.value24();
      Fx = some ? gx + Fx : gx;
      Fy = some ? gy + Fy : gy;
      Fz = some ? gz + Fz : gz;
    }
    f[3 * (int64_t)i + 0] = Fx;
    f[3 * (int64_t)i + 1] = Fy;
    f[3 * (int64_t)i + 2] = Fz;
  }
}

template <int T>
void launch_na_force_fixed(unsigned char* base, const NaParams& p, const double* x, double* f, cudaStream_t s) {
  k_na_force_fixed<T><<<(unsigned)(((int64_t)p.n * T + kNaBlock - 1) / kNaBlock), kNaBlock, 0, s>>>(base, p, x, f);
}

std::mutex g_na_mu;
unsigned char* g_na_addr[kNaMaxDevices] = {};

// Device address of the scratch array on the current device (looked up once).
int na_scratch(unsigned char** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    set_error(std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    return MD_ERR_CUDA;
  }
  if (dev < 0 || dev >= kNaMaxDevices) {
    set_error("device ordinal out of range for md_forces_noalloc");
    return MD_ERR_ARG;
  }
  std::lock_guard<std::mutex> lk(g_na_mu);
  if (!g_na_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      set_error(std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      return MD_ERR_CUDA;
    }
    g_na_addr[dev] = (unsigned char*)p;
  }
  *out = g_na_addr[dev];
  return MD_OK;
}

}  // namespace
}  // namespace ljmd

extern "C" int md_forces_noalloc(const double* x_dev, int64_t N, double box_L, double rc,
                                 double* f_dev, void* stream) {
  using namespace ljmd;
  set_error("");
  if (!x_dev || !f_dev) {
    set_error("null device array");
    return MD_ERR_ARG;
  }
  if (N < 1 || N > kNaMaxN) {
    set_error("md_forces_noalloc: N must be in [1, 65536] (fixed scratch size)");
    return MD_ERR_ARG;
  }
  if (!(rc > 0.0) || !std::isfinite(rc) || !(box_L > 2.0 * rc) || !(box_L <= 10000.0)) {
    set_error("md_forces_noalloc: need rc > 0 and 2 rc < L <= 10000");
    return MD_ERR_ARG;
  }
  unsigned char* base = nullptr;
  int r = na_scratch(&base);
  if (r != MD_OK) return r;
  NaParams p;
  p.L = box_L;
  p.n = (int)N;
  // cells per axis, floor(L / rc), clamped in double before the conversion (L / rc
  // can exceed the int range); lowered by one where rounding could make a cell
  // narrower than rc, and at most 32 (coarser cells stay valid: side > rc)
  const double q = std::floor(box_L / rc);
  int nc = q > 33.0 ? 33 : (int)q;
  if (nc >= 1 && box_L / nc < rc * (1.0 + 1e-9)) nc -= 1;
  if (nc > 32) nc = 32;
  p.nc = nc >= 3 ? nc : 1;
  p.inv_cs = (double)p.nc / box_L;
  p.rc2 = rc * rc;
  const double irc2 = 1.0 / p.rc2, irc6 = irc2 * irc2 * irc2;
  p.c2x8 = 8.0 * (6.0 * irc6 * irc6 * irc2 - 3.0 * irc6 * irc2);
  const int ncell = p.nc * p.nc * p.nc;
  cudaStream_t s = (cudaStream_t)stream;
  const unsigned blocks = (unsigned)((N + 255) / 256);
  k_na_clear<<<(unsigned)((ncell + 255) / 256), 256, 0, s>>>(base, ncell);
  k_na_bin<<<blocks, 256, 0, s>>>(base, p, x_dev);
  k_na_scan<<<1, 1024, 0, s>>>(base, ncell);
  k_na_scatter<<<blocks, 256, 0, s>>>(base, p);
  // Fixed point: cutoffs in its range and cells narrower than 4, so that no candidate is
  // 8 or more away on any axis (positions are kept modulo 16).
  if (p.nc > 1 && rc <= kFixMaxRc && box_L / p.nc < 3.99) {
    p.Lfix = fix_host(box_L);
    p.rc2fix = (long long)std::llrint(std::ldexp(p.rc2, 56));
    p.c2fix = fix_c2(p.c2x8 / 8.0, p.rc2);
    // the high words' separations err by less than 3 units of 2^-28 per axis (2e-8 in all),
    // which counts for cutoffs below 0.004; their float r^2 by a few parts in 1e7
    const double rq = rc + 5.9604644775390625e-08;
    p.rc2q = (float)(std::ldexp(rq * rq, 56) * (1.0 + 1e-5));
    k_na_rank<true><<<blocks, 256, 0, s>>>(base, p, x_dev);
    // threads per particle: enough to fill the GPU
    if (N <= 2432) launch_na_force_fixed<32>(base, p, x_dev, f_dev, s);
    else if (N <= 19456) launch_na_force_fixed<8>(base, p, x_dev, f_dev, s);
    else launch_na_force_fixed<4>(base, p, x_dev, f_dev, s);
  } else {
    k_na_rank<false><<<blocks, 256, 0, s>>>(base, p, x_dev);
    k_na_force<<<blocks, 256, 0, s>>>(base, p, x_dev, f_dev);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error(std::string("md_forces_noalloc launch: ") + cudaGetErrorString(e));
    return MD_ERR_CUDA;
  }
  return MD_OK;
}
