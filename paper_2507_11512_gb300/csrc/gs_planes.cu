// Gauss-Seidel sweeps on the operator evaluated straight from the grid, for one
// right-hand side and for R-vectors: a symmetric sweep in three launches by
// planes, and one launch per colour where planes do not fit.
//
// See stencil.cuh for what they read and why their values equal the ELL
// kernels' bit for bit.

#include <algorithm>
#include <type_traits>

#include "stencil.cuh"

namespace hpg {

// One colour phase (Sec. 3.2.1), one point per thread, in place: what a sweep
// falls back to where an x-line is too long for gs_plane_kernel's shared
// memory, and beside the TMA-tiled phases (HPG_OPT_GS_HALO).  from_zero: only
// neighbours of a lower colour count (first forward sweep from z = 0).
template <typename T>
__global__ void __launch_bounds__(256)
gs_colour_kernel(const __grid_constant__ SGeom g, const __grid_constant__ Coef<T> c, int colour,
                 int from_zero, const T* r, const T* diag, T* z) {
  pdl_trigger();
  pdl_wait();
  const unsigned p = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned row = g.off[colour] + p;
  if (row >= g.end[colour]) return;
  if (p >= g.cnt[colour]) {   // padding row: identity
    const T v = ld_dep(r + row);
    z[row] = from_zero ? v : fma(T(-0.0), ld_dep(z + row), v);
    return;
  }
  const int px = colour_parity_x(colour), py = colour_parity_y(colour),
            pz = colour_parity_z(colour);
  const unsigned w = px ? g.wo : g.we, hl = py ? g.ho : g.he;
  const int e = (int)(p % w);
  const int j = 2 * (int)(p / w % hl) + py, k = 2 * (int)(p / w / hl) + pz;
  const int i = 2 * (e / g.R) + px;
  T acc = ld_dep(r + row);
#pragma unroll
  for (int q = 0; q < kSlots; ++q) {
    const int s = gs_order(q);
    const int dx = s % 3 - 1, dy = (s / 3) % 3 - 1, dz = s / 9 - 1;
    if (s == kCentre) continue;
    const int nc = colour ^ ((dx & 1) | ((dy & 1) << 1) | ((dz & 1) << 2));
    const bool in = (unsigned)(i + dx) < (unsigned)g.nx && (unsigned)(j + dy) < (unsigned)g.ny &&
                    (unsigned)(k + dz) < (unsigned)g.nz && !(from_zero && nc > colour);
    T v = T(0);
    if (in) v = ld_dep(z + line_base(g, px ^ (dx & 1), j + dy, k + dz) + e +
                       ((px + dx) >> 1) * g.R);
    acc = fma(-c.a[dx + dy + dz + 3], v, acc);
  }
  if (!from_zero && on_boundary(g, i, j, k)) acc = fma(T(0), ld_dep(z + row), acc);
  z[row] = acc / (diag ? diag[row / (unsigned)g.R] : (T)kDiag);
}

// The symmetric sweep by planes.  Points of one z parity form whole planes,
// and two planes of the same parity never touch, so the colours 0..3 of a
// forward sweep (the odd planes) need nothing from each other's planes:
// one launch runs them all, plane by plane, and so
//   kOddFwd   colours 0 1 2 3          on the odd planes
//   kEven     colours 4 5 6 7 6 5 4    on the even planes
//   kOddBwd   colours 3 2 1 0          on the odd planes
// is a whole symmetric sweep (15 phases) in 3 launches.  The 18 products with
// the two planes above and below, constant meanwhile, are formed once per
// point (streamed in lines, neighbour lines reused in registers) and kept in
// shared memory; a phase then only adds the 8 products of its own plane, from
// shared memory.
//
// A cluster of `cs` CTAs shares a plane, each owning `lines` x-lines of it.
// A CTA recomputes the one to three lines beyond its own that its last phases
// need, from old values it loads itself, so CTAs exchange nothing; the only
// hazard is that they update z in place, and one cluster barrier -- all old
// values loaded before the first store -- settles it, hidden behind the
// streamed products.
enum PlaneKind { kOddFwd = 0, kEven = 1, kOddBwd = 2 };

struct PlanePlan {
  int lines;    // x-lines per CTA (even)
  int cs;       // CTAs per plane (cluster size)
  int bx, by;   // threads along x, lines in flight
  size_t smem;
};

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

constexpr int kPlaneThreads = 512;

template <typename T, int KIND, bool ZERO>
__global__ void __launch_bounds__(kPlaneThreads, sizeof(T) == 4 ? 2 : 1)
gs_plane_kernel(const __grid_constant__ SGeom g, const __grid_constant__ Coef<T> c,
                const __grid_constant__ PlanePlan pl, const T* r, const T* diag, T* z,
                int c0_done) {
  extern __shared__ __align__(16) unsigned char plane_smem[];
  const int R = g.R, we = g.we, wo = g.wo;
  const int pitch = we + wo + 4 * R;      // a line: [R zeros | even | R zeros][R | odd | R]
  const int oddp = we + 3 * R;            // first odd element of a line
  T* sz = reinterpret_cast<T*>(plane_smem);          // z of lines a-2 ..
  T* sp = sz + (pl.lines + 5) * pitch;               // r minus the outer planes, lines a-1 ..
  T* sd = sp + (pl.lines + 3) * (we + wo);           // diagonal (only with diag)
  const int rank = (int)(blockIdx.x % (unsigned)pl.cs);
  const int k = 2 * (int)(blockIdx.x / (unsigned)pl.cs) + (KIND == kEven ? 0 : 1);
  const int a = rank * pl.lines, b = min(a + pl.lines, g.ny);
  const int tx = threadIdx.x % pl.bx;
  const int ty0 = threadIdx.x / pl.bx;
  const int ty = ty0 < pl.by ? ty0 : (1 << 24);      // threads past the last line row idle
  pdl_trigger();
  pdl_wait();

  // old values of the own plane (zero outside the grid, and before they are
  // first computed in a sweep from zero)
  for (int q = threadIdx.x; q < (pl.lines + 5) * R; q += blockDim.x) {
    T* ln = sz + q / R * pitch + q % R;
    ln[0] = T(0);
    ln[R + we] = T(0);
    ln[2 * R + we] = T(0);
    ln[3 * R + we + wo] = T(0);
  }
  for (int l = ty; l < pl.lines + 5; l += pl.by) {
    const int j = a - 2 + l;
    // lines a-2..b (forward odd planes), a-2..b+2 (even), a-1..b+1 (backward)
    const bool in = j >= (KIND == kOddBwd ? max(a - 1, 0) : 0) && j < g.ny &&
                    j <= b + (KIND == kOddFwd ? 0 : KIND == kEven ? 2 : 1) &&
                    (!ZERO || (KIND == kOddFwd && c0_done && (j & 1)));
    const T* ev = in ? z + line_base(g, 0, j, k) : z;
    const T* od = in ? z + line_base(g, 1, j, k) : z;
    T* ln = sz + l * pitch;
    for (int e = tx; e < we; e += pl.bx) ln[R + e] = in && !ZERO ? ld_dep(ev + e) : T(0);
    for (int e = tx; e < wo; e += pl.bx) ln[oddp + e] = in ? ld_dep(od + e) : T(0);
  }
  __syncwarp();
  if (pl.cs > 1) cluster_arrive();

  // r minus the products with the planes k-1 and k+1
  {
    const int plo = KIND == kOddBwd ? a : max(a - 1, 0);
    const int phi = min(KIND == kEven ? b + 1 : KIND == kOddBwd ? b : b - 1, g.ny - 1);
    const int chunk = (phi - plo + pl.by) / pl.by;
    const int j0 = ty < pl.by ? plo + ty * chunk : g.ny;
    const int j1 = min(j0 + chunk - 1, phi);
    for (int e = tx; e < we && j0 <= j1; e += pl.bx) {
      LinePts<T> lo[3], up[3];
      if (!(ZERO && KIND == kOddFwd)) {
        lo[1] = load_line(z, g, j0 - 1, k - 1, e);
        up[1] = load_line(z, g, j0 - 1, k + 1, e);
        lo[2] = load_line(z, g, j0, k - 1, e);
        up[2] = load_line(z, g, j0, k + 1, e);
      }
      for (int j = j0; j <= j1; ++j) {
        const unsigned pe = line_base(g, 0, j, k) + e, po = line_base(g, 1, j, k) + e;
        T ae = ld_dep(r + pe), ao = e < wo ? ld_dep(r + po) : T(0);
        T* sl = sp + (j - (a - 1)) * (we + wo);
        if (diag) {
          T* dl = sd + (j - (a - 1)) * (we + wo);
          dl[e] = diag[pe / (unsigned)R];
          if (e < wo) dl[we + e] = diag[po / (unsigned)R];
        }
        if (!(ZERO && KIND == kOddFwd)) {
          lo[0] = lo[1];
          lo[1] = lo[2];
          lo[2] = load_line(z, g, j + 1, k - 1, e);
          up[0] = up[1];
          up[1] = up[2];
          up[2] = load_line(z, g, j + 1, k + 1, e);
#pragma unroll
          for (int dy = -1; dy <= 1; ++dy) {
            const LinePts<T>& p = lo[dy + 1];
            ae = line_sum<T, -1>(c, dy - 1, p.l, p.e, p.o, ae);
            ao = line_sum<T, -1>(c, dy - 1, p.e, p.o, p.r, ao);
          }
#pragma unroll
          for (int dy = -1; dy <= 1; ++dy) {
            const LinePts<T>& p = up[dy + 1];
            ae = line_sum<T, -1>(c, dy + 1, p.l, p.e, p.o, ae);
            ao = line_sum<T, -1>(c, dy + 1, p.e, p.o, p.r, ao);
          }
        }
        sl[e] = ae;
        if (e < wo) sl[we + e] = ao;
      }
    }
  }
  __syncwarp();
  if (pl.cs > 1) cluster_wait();
  __syncthreads();

  // one phase: points of x parity XP on the lines lo, lo + 2, .. <= hi; the
  // last update of an own line goes to memory
  auto phase = [&](auto xp, int lo, int hi, bool store) {
    constexpr int XP = decltype(xp)::value;
    const int w = XP ? wo : we;
    for (int j = lo + 2 * ty; j <= hi; j += 2 * pl.by) {
      T* ln = sz + (j - (a - 2)) * pitch;
      const T* su = sp + (j - (a - 1)) * (we + wo) + (XP ? we : 0);
      const bool edge = j == 0 || j == g.ny - 1 || k == 0 || k == g.nz - 1;
      T* out = z + line_base(g, XP, j, k);
      const bool st = store && j >= a && j < b;
      for (int e = tx; e < w; e += pl.bx) {
        // offsets of x-1, x, x+1 in a line
        const int m = (XP ? oddp : R) + e;
        const int xl = XP ? R + e : oddp + e - R, xr = XP ? R + e + R : oddp + e;
        T acc = su[e];
        acc = line_sum<T, -1>(c, -1, ln[xl - pitch], ln[m - pitch], ln[xr - pitch], acc);
        acc = fma(-c.a[2], ln[xl], acc);
        acc = fma(-c.a[4], ln[xr], acc);
        acc = line_sum<T, -1>(c, 1, ln[xl + pitch], ln[m + pitch], ln[xr + pitch], acc);
        const int i = 2 * (e / R) + XP;
        if (edge || i == 0 || i == g.nx - 1) acc = fma(T(0), ln[m], acc);
        acc = diag ? acc / sd[(j - (a - 1)) * (we + wo) + (XP ? we : 0) + e] : acc / (T)kDiag;
        ln[m] = acc;
        if (st) out[e] = acc;
      }
    }
    __syncthreads();
  };
  using Even = std::integral_constant<int, 0>;
  using Odd = std::integral_constant<int, 1>;
  const int top = g.ny - 1;
  if (KIND == kOddFwd) {
    const int lo = a > 0 ? a - 1 : 1;   // odd lines a-1 .. b-1
    if (!c0_done) phase(Odd(), lo, b - 1, true);
    phase(Even(), lo, b - 1, true);
    phase(Odd(), a, b - 1, true);
    phase(Even(), a, b - 1, true);
  } else if (KIND == kEven) {
    const int lo = a > 0 ? a - 1 : 1;
    phase(Odd(), lo, min(b + 1, top), false);
    phase(Even(), lo, min(b + 1, top), false);
    phase(Odd(), a, min(b, top), false);
    phase(Even(), a, min(b, top), true);
    phase(Odd(), a, min(b, top), true);
    phase(Even(), a + 1, b - 1, true);
    phase(Odd(), a + 1, b - 1, true);
  } else {
    phase(Even(), a, min(b, top), true);
    phase(Odd(), a, min(b, top), true);
    phase(Even(), a + 1, b - 1, true);
    phase(Odd(), a + 1, b - 1, true);
  }
  // padding rows (identity) of these planes' colours
  if (blockIdx.x == 0) {
    for (int q = 0; q < 4; ++q) {
      const int cc = (KIND == kEven ? 4 : 0) + q;
      if (c0_done && ZERO && cc == 0) continue;
      for (unsigned p = g.off[cc] + g.cnt[cc] + threadIdx.x; p < g.end[cc]; p += blockDim.x) {
        const T v = ld_dep(r + p);
        z[p] = ZERO ? v : fma(T(-0.0), ld_dep(z + p), v);
      }
    }
  }
}

// Shared memory of a plane CTA with `lines` own lines.
template <typename T>
static size_t plane_smem(const SGeom& g, int lines, bool diag) {
  const size_t row = (size_t)g.we + g.wo;
  return sizeof(T) * ((lines + 5) * (row + 4 * g.R) + (lines + 3) * row * (diag ? 2 : 1));
}

constexpr size_t kMaxPlaneSmem = 227u << 10;
constexpr int kMaxPlaneCtas = 8;   // portable cluster size

// How a level's planes are split: cs CTAs per plane so that about two CTAs
// per SM are busy, with at least 8 lines each (a CTA recomputes up to 3 more),
// more if a CTA's lines would not fit shared memory.  False: no split fits.
template <typename T>
static bool plane_plan(const SGeom& g, int num_sms, bool diag, PlanePlan* out) {
  const int planes = std::max(g.de, 1);
  int cs = 1;
  auto lines_for = [&](int n) { return std::max(2, ((g.ny + n - 1) / n + 1) / 2 * 2); };
  while (cs < kMaxPlaneCtas && planes * (cs + 1) <= 2 * num_sms && lines_for(cs + 1) >= 8) ++cs;
  while (cs <= kMaxPlaneCtas && plane_smem<T>(g, lines_for(cs), diag) > kMaxPlaneSmem) ++cs;
  if (cs > kMaxPlaneCtas) return false;
  PlanePlan p;
  p.lines = lines_for(cs);
  p.cs = (g.ny + p.lines - 1) / p.lines;
  const int pieces = (g.we + 127) / 128;
  p.bx = (g.we + pieces - 1) / pieces;
  p.by = std::max(1, std::min(kPlaneThreads / p.bx, p.lines + 3));
  p.smem = plane_smem<T>(g, p.lines, diag);
  *out = p;
  return true;
}

template <typename T, int KIND, bool ZERO>
static cudaError_t plane_launch(hpg_problem* h, const SGeom& g, const PlanePlan& pl, const T* r,
                                const T* diag, T* z, int c0_done, cudaStream_t s) {
  auto kern = gs_plane_kernel<T, KIND, ZERO>;
  if (pl.smem > (48u << 10)) {
    const cudaError_t e = cudaFuncSetAttribute(
        kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxPlaneSmem);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((KIND == kEven ? g.de : g.dO) * pl.cs));
  cfg.blockDim = dim3((unsigned)((pl.bx * pl.by + 31) / 32 * 32));
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (pl.cs > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = (unsigned)pl.cs;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
  }
  if (h->pdl_enabled && h->pdl_next && !h->profiling) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, kern, g, make_coef<T>(h->beta), pl, r, diag, z, c0_done);
}

template <typename T>
static int colour_phase_t(hpg_problem* h, int level, int R, int colour, bool from_zero,
                          const T* r, T* z, cudaStream_t s) {
  const Level& L = h->lev[level];
  const SGeom g = make_sgeom(L.g, R);
  const unsigned n = g.end[colour] - g.off[colour];
  if (n == 0) return HPG_OK;
  const int nslots = __builtin_popcount(gs_slot_mask(colour, from_zero)) - 1;
  return launch(h, K_GS, level, sizeof(T) == 8 ? HPG_FP64 : HPG_FP32,
                L.cnt[colour] * (2.0 + nslots / 26.0) * R * sizeof(T), s, "gs_colour_kernel",
                [&] {
                  return kl(h, gs_colour_kernel<T>, grid_for(n, 256), 256, s, g,
                            make_coef<T>(h->beta), colour, (int)from_zero, r, level_diag<T>(L),
                            z);
                });
}
int stencil_colour_phase(hpg_problem* h, int level, int R, int colour, bool from_zero,
                         const float* r, float* z, cudaStream_t s) {
  return colour_phase_t<float>(h, level, R, colour, from_zero, r, z, s);
}
int stencil_colour_phase(hpg_problem* h, int level, int R, int colour, bool from_zero,
                         const double* r, double* z, cudaStream_t s) {
  return colour_phase_t<double>(h, level, R, colour, from_zero, r, z, s);
}

// One symmetric sweep; c0_done: z already holds colour 0's first phase.
template <typename T>
static int symgs_t(hpg_problem* h, int level, int R, const T* r, T* z, bool from_zero,
                   bool c0_done, cudaStream_t s) {
  const Level& L = h->lev[level];
  const SGeom g = make_sgeom(L.g, R);
  const T* diag = level_diag<T>(L);
  int rc;
  PlanePlan pl;
  if (!plane_plan<T>(g, h->num_sms, diag != nullptr, &pl)) {
    for (int c = c0_done ? 1 : 0; c < kColours; ++c)
      if ((rc = stencil_colour_phase(h, level, R, c, from_zero, r, z, s))) return rc;
    for (int c = kColours - 2; c >= 0; --c)
      if ((rc = stencil_colour_phase(h, level, R, c, false, r, z, s))) return rc;
    return HPG_OK;
  }
  const int prec = sizeof(T) == 8 ? HPG_FP64 : HPG_FP32;
  auto phases = [&](int lo, int hi) {   // non-empty colours lo..hi
    int n = 0;
    for (int c = lo; c <= hi; ++c) n += L.cnt[c] > 0;
    return n;
  };
  double half[2] = {0.0, 0.0};   // elements of the odd and the even planes
  for (int c = 0; c < kColours; ++c) half[c >> 2] += (double)L.cnt[c] * R;
  const double all = half[0] + half[1], sv = sizeof(T);
  if (g.dO > 0) {
    // r read, z written; not from zero: all of z read
    rc = launch(h, K_GS, level, prec, (half[0] * 2 + (from_zero ? 0.0 : all)) * sv, s,
                "gs_plane_kernel", [&] {
                  return from_zero ? plane_launch<T, kOddFwd, true>(h, g, pl, r, diag, z, c0_done, s)
                                   : plane_launch<T, kOddFwd, false>(h, g, pl, r, diag, z, c0_done, s);
                }, phases(c0_done ? 1 : 0, 3));
    if (rc) return rc;
  }
  rc = launch(h, K_GS, level, prec, (half[1] * 2 + (from_zero ? half[0] : all)) * sv, s,
              "gs_plane_kernel", [&] {
                return from_zero ? plane_launch<T, kEven, true>(h, g, pl, r, diag, z, 0, s)
                                 : plane_launch<T, kEven, false>(h, g, pl, r, diag, z, 0, s);
              }, phases(4, 7) + phases(4, 6));
  if (rc || g.dO == 0) return rc;
  return launch(h, K_GS, level, prec, (half[0] * 2 + all) * sv, s, "gs_plane_kernel",
                [&] { return plane_launch<T, kOddBwd, false>(h, g, pl, r, diag, z, 0, s); },
                phases(0, 3));
}
int stencil_symgs(hpg_problem* h, int level, int R, const float* r, float* z, bool from_zero,
                  bool c0_done, cudaStream_t s) {
  return symgs_t<float>(h, level, R, r, z, from_zero, c0_done, s);
}
int stencil_symgs(hpg_problem* h, int level, int R, const double* r, double* z, bool from_zero,
                  bool c0_done, cudaStream_t s) {
  return symgs_t<double>(h, level, R, r, z, from_zero, c0_done, s);
}

}  // namespace hpg
