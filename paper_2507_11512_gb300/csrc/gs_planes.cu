// Gauss-Seidel sweeps on the operator evaluated straight from the grid, for one
// right-hand side and for R-vectors: a symmetric sweep in three launches by
// planes, and one launch per colour where planes do not fit.
//
// See stencil.cuh for what they read and why their values equal the ELL
// kernels' bit for bit.

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "stencil.cuh"

namespace hpg {

// One colour phase (Sec. 3.2.1), V consecutive elements of a line per thread (V
// divides R, so that neighbour groups are aligned), in place: FP64 sweeps of larger
// levels and levels whose planes do not fit (see symgs_t), and phases beside the
// TMA-tiled ones (HPG_OPT_GS_HALO).  Small phases are bound by the chain of wait, loads,
// products and division, so positions and line addresses are formed before the wait,
// from eight bases and fixed steps, and no load waits for another; large FP32 ones by
// instruction issue; FP64 by the FP64 unit (29 operations a point, 16 cycles a warp
// instruction and SM), which small blocks spread evenly.  One sweep, against a
// kernel that found each neighbour's line by itself after the wait and read the own entry
// of boundary points last: FP32 2000 x 4 x 4 47 -> 25 us, 400 x 400 x 40 373 -> 165; FP64
// 2000 x 4 x 4 54 -> 38, 112^3 218 -> 195, 160^3 511 -> 478; 256 x 256 x 8 with eight
// right-hand sides, V-cycle 634 -> 254 (two elements a thread; four held too few loads in
// flight, 309).  MC = -1: all
// neighbours; MC = 0..7: the phase of colour MC in the first forward sweep from
// z = 0, where only neighbours of a lower colour count (the set is fixed at compile
// time).
template <typename T, int V, int MC>
__global__ void __launch_bounds__(256)
gs_colour_kernel(const __grid_constant__ ColourPlan g, const __grid_constant__ Coef<T> c,
                 const T* r, const T* diag, T* z) {
  constexpr unsigned kMask = MC < 0 ? (1u << kSlots) - 1u : gs_slot_mask(MC, true);
  using P = typename VecOf<T, V>::type;
  if (g.early) pdl_trigger();
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned p = t * V, row = g.off + p;
  if (row >= g.end) return;
  if (p >= g.cnt) {   // padding row: identity
    pdl_wait();
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const T rv = ld_dep(r + row + v);
      z[row + v] = MC >= 0 ? rv : fma(T(-0.0), ld_dep(z + row + v), rv);
    }
    return;
  }
  const ColourPlace at(g, t, V);
  const bool edge = at.edge();
  const T dg = diag ? diag[row >> g.rshift] : T(0);
  pdl_wait();
  T x[kSlots][V], u[V];
#pragma unroll
  for (int s = 0; s < kSlots; ++s) {
#pragma unroll
    for (int v = 0; v < V; ++v) x[s][v] = T(0);
    if (s == kCentre ? MC >= 0 : !((kMask >> s) & 1u)) continue;
    if (s == kCentre ? edge : at.in(s)) unpack(ld_dep(reinterpret_cast<const P*>(z + at.at(g, s))), x[s]);
  }
  unpack(ld_dep(reinterpret_cast<const P*>(r + row)), u);
#pragma unroll
  for (int s = 0; s < kSlots; ++s)
    if (s != kCentre && ((kMask >> s) & 1u)) {
#pragma unroll
      for (int v = 0; v < V; ++v)
        u[v] = fma(-c.a[s % 3 - 1 + (s / 3) % 3 - 1 + s / 9 - 1 + 3], x[s][v], u[v]);
    }
  if (MC < 0 && edge) {
#pragma unroll
    for (int v = 0; v < V; ++v) pad_slot(x[kCentre][v], u[v]);
  }
  if (diag) {
#pragma unroll
    for (int v = 0; v < V; ++v) u[v] = u[v] / dg;
  } else {
    div_diag<T, V>(u);
  }
  bool all[V];
#pragma unroll
  for (int v = 0; v < V; ++v) all[v] = true;
  store_elems<T, V, true>(z + row, all, u);
}

template <typename T>
using ColourFn = void (*)(const ColourPlan, const Coef<T>, const T*, const T*, T*);
template <typename T, int V> static ColourFn<T> colour_fn(int colour, bool from_zero) {
  if (!from_zero) return gs_colour_kernel<T, V, -1>;
  switch (colour) {
    case 0: return gs_colour_kernel<T, V, 0>;
    case 1: return gs_colour_kernel<T, V, 1>;
    case 2: return gs_colour_kernel<T, V, 2>;
    case 3: return gs_colour_kernel<T, V, 3>;
    case 4: return gs_colour_kernel<T, V, 4>;
    case 5: return gs_colour_kernel<T, V, 5>;
    case 6: return gs_colour_kernel<T, V, 6>;
    default: return gs_colour_kernel<T, V, 7>;
  }
}

// The symmetric sweep by planes.  Points of one z parity form whole planes,
// and two planes of the same parity never touch, so the colours 0..3 of a
// forward sweep (the odd planes) need nothing from each other's planes:
// one launch runs them all, plane by plane, and so
//   kOddFwd   colours 0 1 2 3          on the odd planes
//   kEven     colours 4 5 6 7 6 5 4    on the even planes
//   kOddBwd   colours 3 2 1 0          on the odd planes
// is a whole symmetric sweep (15 phases) in 3 launches.  A CTA copies its
// lines of the plane and of the two planes beside it (constant meanwhile) into
// shared memory, all at once, and every phase runs from there.
// The products of a row keep slot order -- plane below, own plane, plane above --
// so values equal the one-launch-per-colour sweep's bit for bit.
//
// A cluster of `cs` CTAs shares a plane, each owning `lines` x-lines of it.
// A CTA recomputes the one to three lines beyond its own that its last phases
// need, from old values it loads itself, so CTAs exchange nothing; the only
// hazard is that they update z in place, and one cluster barrier -- all old
// values loaded before the first store -- settles it: a CTA arrives once its
// loads are done and waits only before it stores, after its last phase.
//
// Large grids are bound by the vectors' traffic and by instruction issue (R
// and the loads' offsets are compile-time, two or four FP32 elements share loads and
// addresses for that reason), FP64 by the FP64 rate; small ones by the chain of
// load, phases and store.
// One sweep on GB300, stored matrix with a launch per colour -> this: FP32 64^3 39
// -> 13 us, 128^3 139 -> 30 us, 320^3 2.1 ms -> 495 us; FP64 64^3 66 -> 48 us.  Where
// whole planes leave SMs without work the sweep goes by colours (by_colours).
enum PlaneKind { kOddFwd = 0, kEven = 1, kOddBwd = 2 };

struct PlanePlan {
  int lines;    // x-lines per CTA (even)
  int cs;       // CTAs per plane (cluster size)
  int bx, by;   // threads along x, lines in flight (even)
  int early;    // whether the next kernel may start while this one runs
  size_t smem;
};

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Asynchronous copy of B bytes global -> shared, or zeros where !in (src is not
// read then), completed by copy_wait().
template <int B> __device__ __forceinline__ void copy_async(void* dst, const void* src, bool in) {
  if constexpr (B == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src),
                 "r"(in ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_addr(dst)), "l"(src),
                 "n"(B), "r"(in ? B : 0) : "memory");
}
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Threads of a plane CTA, at most (a line's element groups must fit).  At the kernels'
// 64 to 80 registers one such CTA fits an SM; plans for two take half the threads.
constexpr int kPlaneThreads = 768;
// Shared-memory layout of a CTA: z of the lines a-2 .. b+2 of the planes k-1, k
// and k+1, each line as
//   [pad | even part | pad | odd part | pad]   (pads zero, parts rounded to V)
template <int R, int V> struct PlaneLayout {
  int part, pitch, odd;
  __host__ __device__ explicit PlaneLayout(const SGeom& g) {
    part = (g.we + V - 1) / V * V;
    odd = 2 * pad() + part;
    pitch = 2 * part + 3 * pad();
  }
  static __host__ __device__ constexpr int pad() { return R > V ? R : V; }
  __host__ __device__ size_t elems(int lines) const {
    return (size_t)(lines + 5) * pitch * 3;
  }
};

template <typename T, int V>
__device__ __forceinline__ void lds(const T* p, T (&a)[V]) {
  unpack(*reinterpret_cast<const typename VecOf<T, V>::type*>(p), a);
}

// What a thread's elements touch on one line in shared memory.
template <typename T, int R, int V>
__device__ __forceinline__ LinePts<T, V> smem_line(const T* ev, const T* od) {
  LinePts<T, V> p;
  lds<T, V>(ev, p.e);
  lds<T, V>(od, p.o);
  if constexpr (R % V == 0) {
    lds<T, V>(od - R, p.l);
    lds<T, V>(ev + R, p.r);
  } else {
    p.l[0] = od[-1];
    p.r[V - 1] = ev[V];
#pragma unroll
    for (int v = 1; v < V; ++v) {
      p.l[v] = p.o[v - 1];
      p.r[v - 1] = p.e[v];
    }
  }
  return p;
}

// u minus the products of one line in shared memory, for the points of x parity
// XO (R a multiple of V).
template <typename T, int R, int V, bool XO>
__device__ __forceinline__ void half_line(const Coef<T>& c, int dyz, const T* ev, const T* od,
                                          T (&u)[V]) {
  T l[V], q[V], r[V];
  lds<T, V>(XO ? ev : od - R, l);
  lds<T, V>(XO ? od : ev, q);
  lds<T, V>(XO ? ev + R : od, r);
#pragma unroll
  for (int v = 0; v < V; ++v)
    u[v] = fma(-c.a[dyz + 4], r[v], fma(-c.a[dyz + 3], q[v], fma(-c.a[dyz + 2], l[v], u[v])));
}

template <typename T, int R, int V, bool VEC, int KIND, bool ZERO>
__global__ void __launch_bounds__(kPlaneThreads)
gs_plane_kernel(const __grid_constant__ SGeom g, const __grid_constant__ Coef<T> c,
                const __grid_constant__ PlanePlan pl, const T* r, const T* diag, T* z,
                int c0_done) {
  extern __shared__ __align__(16) unsigned char plane_smem[];
  const PlaneLayout<R, V> lay(g);
  const int we = g.we, wo = g.wo;
  const int slab = (pl.lines + 5) * lay.pitch;
  T* const sz = reinterpret_cast<T*>(plane_smem) + slab;   // plane k; k-1 before, k+1 after
  constexpr bool outer = !(ZERO && KIND == kOddFwd);       // the planes beside are not zero
  // the line and the plane after in registers for both x parities; four-element
  // R-vector groups (64 registers of them) read them again instead
  constexpr bool kHold = R % V != 0 || V < 4;
  const int rank = (int)(blockIdx.x % (unsigned)pl.cs);
  const int k = 2 * (int)(blockIdx.x / (unsigned)pl.cs) + (KIND == kEven ? 0 : 1);
  const int a = rank * pl.lines, b = min(a + pl.lines, g.ny);
  const int top = g.ny - 1;
  const int x = (int)(threadIdx.x % (unsigned)pl.bx) * V;
  const int ty0 = (int)(threadIdx.x / (unsigned)pl.bx);
  const int ty = ty0 < pl.by ? ty0 : (1 << 24);      // threads past the last row idle
  const XMask<R, V, VEC> m(g, x);
  if (pl.early) pdl_trigger();
  // zeros around the parts
  {
    constexpr int pad = PlaneLayout<R, V>::pad();
    const int first = outer ? 0 : pl.lines + 5, last = (outer ? 3 : 2) * (pl.lines + 5);
    for (int l = first + (int)threadIdx.x; l < last; l += blockDim.x) {
      T* ln = sz + l * lay.pitch - slab;
#pragma unroll
      for (int e = 0; e < pad; ++e) ln[e] = ln[lay.odd - pad + e] = ln[lay.pitch - pad + e] = T(0);
      if (!VEC)   // parts that are not whole groups
        for (int e = 0; e < V; ++e) ln[lay.odd - pad - 1 - e] = ln[lay.pitch - pad - 1 - e] = T(0);
    }
    if (!VEC) __syncthreads();   // the parts' ends are written below
  }
  pdl_wait();

  // The lines zlo .. zhi of the three planes (zero outside the grid; the own
  // plane's also before they are first computed in a sweep from zero).  by is
  // even, so a thread's lines have one parity and its pointers a fixed step.
  const int zlo = max(KIND == kOddBwd ? a - 1 : a - 2, 0);
  const int zhi = min(KIND == kOddFwd ? b : KIND == kEven ? b + 2 : b + 1, top);
  if (ty < pl.by) {
    const int p = ty & 1;   // a is even: the parity of a - 2 + ty
    const bool in_lo = k > 0, in_up = k + 1 < g.nz;
    const PlanePtr<T> p0(z, g, k, x), p1(z, g, in_lo ? k - 1 : k, x), p2(z, g, in_up ? k + 1 : k, x);
    const bool own_o = !ZERO || (KIND == kOddFwd && c0_done && p);   // from zero: colour 0 at most
    T* le = sz + ty * lay.pitch + lay.pad() + x;
    T* lo = le - lay.pad() + lay.odd;
    constexpr int B = VEC ? V * (int)sizeof(T) : (int)sizeof(T);
    constexpr int N = VEC ? 1 : V;
    for (int l = ty; l < pl.lines + 5; l += pl.by) {
      const int j = a - 2 + l;
      const bool in = j >= zlo && j <= zhi;
      const int oe = in ? (j >> 1) * we : 0, oo = in ? (j >> 1) * wo : 0;
#pragma unroll
      for (int v = 0; v < N; ++v) {
        if (m.e[v]) {
          copy_async<B>(le + v, p0.ev[p] + oe + v, in && !ZERO);
          if (outer) {
            copy_async<B>(le + v - slab, p1.ev[p] + oe + v, in && in_lo);
            copy_async<B>(le + v + slab, p2.ev[p] + oe + v, in && in_up);
          }
        }
        if (VEC || m.o[v]) {   // whole groups: zeros past the end of an odd part
          const bool has = in && m.o[v];
          copy_async<B>(lo + v, p0.od[p] + oo + v, has && own_o);
          if (outer) {
            copy_async<B>(lo + v - slab, p1.od[p] + oo + v, has && in_lo);
            copy_async<B>(lo + v + slab, p2.od[p] + oo + v, has && in_up);
          }
        }
      }
      le += pl.by * lay.pitch;
      lo += pl.by * lay.pitch;
    }
  }
  const PlanePtr<T> pz(z, g, k, x), pr(r, g, k, x);
  // which of the thread's even / odd points lie on an x face of the grid
  unsigned edge_e = 0, edge_o = 0;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    edge_e |= x_edge(g, 0, x + v) ? 1u << v : 0u;
    edge_o |= x_edge(g, 1, x + v) ? 1u << v : 0u;
  }
  const bool edge_k = k == 0 || k == g.nz - 1;
  // r of the next pass's line, loaded a pass ahead
  T re[V] = {}, ro[V] = {};
  auto fetch_r = [&](int j, int hi) {
    if (j <= hi) {
      load_elems<T, V, VEC>(pr.ev[j & 1] + (j >> 1) * we, m.e, re);
      load_elems<T, V, VEC>(pr.od[j & 1] + (j >> 1) * wo, m.o, ro);
    }
  };
  const int olo = a > 0 && KIND != kOddBwd ? a - 1 : a + 1;   // first odd line of the first call
  const int ohi = min(KIND == kEven ? b + 1 : b - 1, top);
  if (KIND == kOddBwd || olo > ohi) fetch_r(a + 2 * ty, min(b, top));   // (no odd line)
  else fetch_r(olo + 2 * ty, ohi);
  copy_wait();
  __syncwarp();
  if (pl.cs > 1) cluster_arrive();
  __syncthreads();

  // Colours of the lines lo, lo + 2, .. <= hi (one line parity), in the order
  // x odd (ODD1), x even, x odd again (ODD2): the products up to the line before,
  // once, then the updates.  nlo, nhi: the lines of the next call.
  auto colours = [&](auto odd1, auto odd2, bool skip, int lo, int hi, int nlo, int nhi) {
    constexpr bool ODD1 = decltype(odd1)::value, ODD2 = decltype(odd2)::value;
    for (int jb = lo; jb <= hi; jb += 2 * pl.by) {
      const int j = jb + 2 * ty;
      const bool on = j <= hi;
      T ae[V], ao[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        ae[v] = re[v];
        ao[v] = ro[v];
      }
      const bool more = jb + 2 * pl.by <= hi;
      fetch_r(more ? j + 2 * pl.by : nlo + 2 * ty, more ? hi : nhi);
      T* le = sz + (on ? j - (a - 2) : 1) * lay.pitch + lay.pad() + x;
      T* lod = le - lay.pad() + lay.odd;
      LinePts<T, V> after, w[3];
      T de[V], dd[V];
      unsigned be = 0, bo = 0;
      if (on) {
        if (diag) {
#pragma unroll
          for (int v = 0; v < V; ++v) {
            de[v] = m.e[v] ? diag[(pr.ev[j & 1] + (j >> 1) * we - r + v) / R] : T(1);
            dd[v] = m.o[v] ? diag[(pr.od[j & 1] + (j >> 1) * wo - r + v) / R] : T(1);
          }
        }
        if (outer) {
#pragma unroll
          for (int u = 0; u < 3; ++u) {   // the lines j - 1, j, j + 1 of plane k - 1
            const int o = (u - 1) * lay.pitch - slab;
            line_sum<T, -1, V>(c, u - 2, smem_line<T, R, V>(le + o, lod + o), ae, ao);
          }
        }
        line_sum<T, -1, V>(c, -1, smem_line<T, R, V>(le - lay.pitch, lod - lay.pitch), ae, ao);
        if (kHold) {
          after = smem_line<T, R, V>(le + lay.pitch, lod + lay.pitch);
          if (outer) {
#pragma unroll
            for (int u = 0; u < 3; ++u) {
              const int o = (u - 1) * lay.pitch + slab;
              w[u] = smem_line<T, R, V>(le + o, lod + o);
            }
          }
        }
        const bool all = edge_k || j == 0 || j == top;
        be = all ? 15u : edge_e;
        bo = all ? 15u : edge_o;
      }
      // x odd: neighbours even[x], even[x + R]; x even: odd[x - R], odd[x]
      auto update = [&](auto xodd) {
        constexpr bool XO = decltype(xodd)::value;
        if (on) {
          T l[V], q[V], u[V];
          T* own = XO ? lod : le;
          if constexpr (XO) {
            lds<T, V>(le, l);
            if constexpr (R % V == 0) {
              lds<T, V>(le + R, q);
            } else {
#pragma unroll
              for (int v = 0; v + 1 < V; ++v) q[v] = l[v + 1];
              q[V - 1] = le[V];
            }
          } else {
            lds<T, V>(lod, q);
            if constexpr (R % V == 0) {
              lds<T, V>(lod - R, l);
            } else {
              l[0] = lod[-1];
#pragma unroll
              for (int v = 1; v < V; ++v) l[v] = q[v - 1];
            }
          }
#pragma unroll
          for (int v = 0; v < V; ++v)
            u[v] = fma(-c.a[4], q[v], fma(-c.a[2], l[v], XO ? ao[v] : ae[v]));
          if (kHold) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
              u[v] = half_sum<T, XO>(c, 1, after, v, u[v]);
              if (outer) {
#pragma unroll
                for (int d = 0; d < 3; ++d) u[v] = half_sum<T, XO>(c, d, w[d], v, u[v]);
              }
            }
          } else {
            half_line<T, R, V, XO>(c, 1, le + lay.pitch, lod + lay.pitch, u);
            if (outer) {
#pragma unroll
              for (int d = 0; d < 3; ++d)
                half_line<T, R, V, XO>(c, d, le + (d - 1) * lay.pitch + slab,
                                       lod + (d - 1) * lay.pitch + slab, u);
            }
          }
          if (XO ? bo : be) {
            T v0[V];
            lds<T, V>(own, v0);
#pragma unroll
            for (int v = 0; v < V; ++v)
              if (((XO ? bo : be) >> v) & 1u) pad_slot(v0[v], u[v]);
          }
          if (diag) {
#pragma unroll
            for (int v = 0; v < V; ++v) u[v] = u[v] / (XO ? dd[v] : de[v]);
          } else {
            div_diag<T, V>(u);
          }
          store_elems<T, V, VEC>(own, XO ? m.o : m.e, u);
        }
        __syncthreads();
      };
      if (ODD1 && !skip) update(std::true_type());
      update(std::false_type());
      if (ODD2) update(std::true_type());
    }
  };
  using Yes = std::true_type;
  using No = std::false_type;
  const int eb = min(b, top), ob = min(b + 1, top);
  if (KIND == kOddFwd) {
    colours(Yes(), No(), c0_done != 0, olo, b - 1, a, b - 1);   // odd lines a-1 .. b-1
    colours(Yes(), No(), false, a, b - 1, 0, -1);
  } else if (KIND == kEven) {
    colours(Yes(), No(), false, olo, ob, a, eb);
    colours(Yes(), Yes(), false, a, eb, a + 1, b - 1);
    colours(No(), Yes(), false, a + 1, b - 1, 0, -1);
  } else {
    colours(No(), Yes(), false, a, eb, a + 1, b - 1);
    colours(No(), Yes(), false, a + 1, b - 1, 0, -1);
  }
  __syncwarp();
  if (pl.cs > 1) cluster_wait();
  {
    for (int j = a + ty; j < b; j += pl.by) {
      const T* ln = sz + (j - (a - 2)) * lay.pitch + x;
      T v[V];
      lds<T, V>(ln + lay.pad(), v);
      store_elems<T, V, VEC>(const_cast<T*>(pz.ev[j & 1]) + (j >> 1) * we, m.e, v);
      lds<T, V>(ln + lay.odd, v);
      store_elems<T, V, VEC>(const_cast<T*>(pz.od[j & 1]) + (j >> 1) * wo, m.o, v);
    }
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

// Shared memory of a plane CTA with `lines` own lines, V elements a thread.
template <typename T, int V>
static size_t plane_smem(const SGeom& g, int lines) {
  const size_t n = g.R == 1   ? PlaneLayout<1, V>(g).elems(lines)
                   : g.R == 2 ? PlaneLayout<2, V>(g).elems(lines)
                   : g.R == 4 ? PlaneLayout<4, V>(g).elems(lines)
                              : PlaneLayout<8, V>(g).elems(lines);
  return sizeof(T) * n;
}

constexpr size_t kMaxPlaneSmem = 227u << 10;
constexpr size_t kPlaneSmemGoal = 112u << 10;   // two CTAs per SM
constexpr int kMaxPlaneCtas = 8;                // portable cluster size

// How a level's planes are split.  FP32: up to 4 CTAs per plane while that makes
// at most two CTAs per SM, with at least 8 lines each (a CTA recomputes up to 3
// more).  FP64, whose time is the busiest SM's FP64 work: the split of up to 5 CTAs
// with the fewest lines on that SM -- one CTA per SM up to 85 % of the SMs (clusters
// do not reach all of them), else whole rounds of two (64^3 sweep 76 -> 48 us against 5
// CTAs throughout).  Up to 8 where a CTA's lines would take more shared memory than
// two CTAs per SM have.  (Measured, one sweep: 128^3 FP32 30 us with 4 CTAs per plane,
// 37 with 3 or 8.)  About 384 threads a CTA, twice that where only one fits an SM.
// The next kernel may start early only after grids that leave most SMs idle:
// otherwise its waiting CTAs take the free places unevenly (96^3 FP64 V-cycle by planes
// 595 us with an early start everywhere, 493 with this rule; 8^3 sweep 11.5 us without
// any, 9.5 with).
// False: a line has more element groups than a CTA threads, or its lines do not
// fit shared memory even so.
template <typename T, int V>
static bool plane_plan(const SGeom& g, int num_sms, PlanePlan* out) {
  const int planes = std::max(g.de, 1);
  int cs = 1;
  auto lines_for = [&](int n) { return std::max(2, ((g.ny + n - 1) / n + 1) / 2 * 2); };
  if (sizeof(T) == 8) {
    double best = 1e30;
    for (int n = 1; n <= 5 && (n == 1 || lines_for(n) >= 8); ++n) {
      const int ctas = planes * n;
      const int rounds = ctas <= num_sms * 0.85 ? 1 : (ctas + 2 * num_sms - 1) / (2 * num_sms) * 2;
      const double cost = rounds * (lines_for(n) + 1.5);
      if (cost < best) {
        best = cost;
        cs = n;
      }
    }
  } else {
    while (cs < 4 && planes * (cs + 1) <= 2 * num_sms && lines_for(cs + 1) >= 8) ++cs;
  }
  while (cs < kMaxPlaneCtas && plane_smem<T, V>(g, lines_for(cs)) > kPlaneSmemGoal) ++cs;
  if (plane_smem<T, V>(g, lines_for(cs)) > kMaxPlaneSmem) return false;
  PlanePlan p;
  p.lines = lines_for(cs);
  p.cs = (g.ny + p.lines - 1) / p.lines;
  p.bx = (g.we + V - 1) / V;
  if (2 * p.bx > kPlaneThreads) return false;
  // a phase has up to lines / 2 + 2 lines
  const int rows = p.lines / 2 + 2;
  p.smem = plane_smem<T, V>(g, p.lines);
  const int threads = p.smem > kPlaneSmemGoal ? kPlaneThreads : kPlaneThreads / 2;
  const int fit = std::max(2, threads / p.bx & ~1);
  const int passes = (rows + fit - 1) / fit;
  p.by = ((rows + passes - 1) / passes + 1) & ~1;   // even (see the copies)
  p.early = planes * p.cs <= num_sms / 4;
  *out = p;
  return true;
}

template <typename T, int R, int V, bool VEC, int KIND, bool ZERO>
static cudaError_t plane_launch_r(hpg_problem* h, const SGeom& g, const PlanePlan& pl, const T* r,
                                  const T* diag, T* z, int c0_done, cudaStream_t s) {
  auto kern = gs_plane_kernel<T, R, V, VEC, KIND, ZERO>;
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

// Elements a thread takes.  FP32 on large levels four where a line's parts and R
// divide by it (they share each load, address and boundary test: 128^3 sweep 43
// -> 32 us), else two (on small levels the longer code costs more than it saves:
// 64^3 23 against 15 us); a line of odd width is read one by one.  FP64 one
// (bound by its FMAs).
template <typename T>
static int plane_elems(const SGeom& g, const T* r, const T* z, bool* vec) {
  *vec = true;
  if (sizeof(T) == 8) return 1;
  const bool large = (double)g.nx * g.ny * g.nz * g.R >= 600000.0;
  if (large && (g.R == 1 || g.R >= 4) && whole_groups<T, 4>(g, r, z)) return 4;
  *vec = whole_groups<T, 2>(g, r, z);
  return 2;
}

template <typename T, int KIND, bool ZERO>
static cudaError_t plane_launch(hpg_problem* h, const SGeom& g, int V, bool vec,
                                const PlanePlan& pl, const T* r, const T* diag, T* z, int c0_done,
                                cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {   // R-vectors are FP32
    if (g.R == 8)
      return V == 4 ? plane_launch_r<T, 8, 4, true, KIND, ZERO>(h, g, pl, r, diag, z, c0_done, s)
                    : plane_launch_r<T, 8, 2, true, KIND, ZERO>(h, g, pl, r, diag, z, c0_done, s);
    if (g.R == 4)
      return V == 4 ? plane_launch_r<T, 4, 4, true, KIND, ZERO>(h, g, pl, r, diag, z, c0_done, s)
                    : plane_launch_r<T, 4, 2, true, KIND, ZERO>(h, g, pl, r, diag, z, c0_done, s);
    if (g.R == 2) return plane_launch_r<T, 2, 2, true, KIND, ZERO>(h, g, pl, r, diag, z, c0_done, s);
    if (V == 4) return plane_launch_r<T, 1, 4, true, KIND, ZERO>(h, g, pl, r, diag, z, c0_done, s);
    if (!vec) return plane_launch_r<T, 1, 2, false, KIND, ZERO>(h, g, pl, r, diag, z, c0_done, s);
    return plane_launch_r<T, 1, 2, true, KIND, ZERO>(h, g, pl, r, diag, z, c0_done, s);
  } else {
    return plane_launch_r<T, 1, 1, true, KIND, ZERO>(h, g, pl, r, diag, z, c0_done, s);
  }
}

// Whether the next phase may start while one of `threads` threads runs.  Its blocks
// then wait in the places that are left, and spread unevenly over the SMs, unless
// the phase is so small that it does not matter or takes every place itself (1024
// FP64 threads an SM at these kernels' registers, 1536 FP32).  One sweep, early /
// not: FP64 40^3 40.6 / 40.9 us, 48^3 43.8 / 43.0, 80^3 135 / 87, 104^3 161 / 157, 112^3
// 195 / 197; FP32 64^3 28.6 / 28.2, 88^3 46 / 39, 112^3 54.7 / 53.8, 120^3 56 / 61.
template <typename T> static int colour_early(long long threads, int num_sms) {
  const long long few = sizeof(T) == 8 ? 80 : 260, full = sizeof(T) == 8 ? 980 : 1350;
  return threads <= few * num_sms || threads >= full * num_sms;
}

template <typename T>
static int colour_phase_t(hpg_problem* h, int level, int R, int colour, bool from_zero,
                          const T* r, T* z, cudaStream_t s) {
  const Level& L = h->lev[level];
  const SGeom g = make_sgeom(L.g, R);
  const unsigned n = g.end[colour] - g.off[colour];
  if (n == 0) return HPG_OK;
  const int nslots = __builtin_popcount(gs_slot_mask(colour, from_zero)) - 1;
  // two elements of an aligned R-vector share loads, addresses and tests
  const int V = R > 1 && (((uintptr_t)r | (uintptr_t)z) & 7u) == 0 ? 2 : 1;
  ColourPlan q = make_colour_plan(
      g, colour, Div31((unsigned)((colour_parity_x(colour) ? g.wo : g.we) / V)),
      Div31((unsigned)(colour_parity_y(colour) ? g.ho : g.he)));
  q.early = colour_early<T>(n / V, h->num_sms);
  return launch(h, K_GS, level, sizeof(T) == 8 ? HPG_FP64 : HPG_FP32,
                L.cnt[colour] * (2.0 + nslots / 26.0) * R * sizeof(T), s, "gs_colour_kernel",
                [&] {
                  const int block = sizeof(T) == 8 ? 64 : 256;
                  ColourFn<T> fn = colour_fn<T, 1>(colour, from_zero);
                  if constexpr (sizeof(T) == 4) {
                    if (V == 2) fn = colour_fn<T, 2>(colour, from_zero);
                  }
                  return kl(h, fn, grid_for(n / V, block), block, s, q, make_coef<T>(h->beta), r,
                            level_diag<T>(L), z);
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

// Whether a sweep takes one launch per colour although its planes fit: where whole
// planes leave SMs without work (few planes, or FP64, whose time is the busiest SM's),
// or lines are so short that a thread's elements are padding.  Both times are
// estimated, in us, from linear fits to 550 sweeps (GB300, 1 to 8 right-hand sides,
// cubes of 12 to 208 and flat, long and thin grids): planes by the busiest SM's elements
// (of the lines a CTA computes, in thousands) and its rounds of lines, colours by
// phases and elements per SM, to 15 % and 6 %.  `least` counts what the host needs to
// launch a phase where that is more.  Planes against colours, one sweep:
// FP64 64^3 48 / 60 us, 72^3 77 / 69, 96^3 150 / 132, 128^3 434 / 263, 200 x 200 x 1 92 / 19,
// 128 x 128 x 8 136 / 43, 64 x 64 x 16 43 / 40, 8 x 1000 x 8 73 / 40; FP32 128^3 31 / 68, 128 x
// 128 x 8 22 / 27, 300 x 300 x 4 47 / 32, 16 x 2000 x 4 44 / 27, 1 x 1000 x 1000 82 / 29.
struct SweepCost { double launch, work, round, phase, element, least; };
template <typename T>
static bool by_colours(const SGeom& g, const Level& L, const PlanePlan& pl, int V, bool vec,
                       int num_sms) {
  const SweepCost c = sizeof(T) == 8 ? SweepCost{4.0, 11.0, 1.0, 2.3, 8.4, 3.3}
                      : g.R == 1     ? SweepCost{3.3, 1.0, 0.25, 1.9, 1.66, 1.9}
                                     : SweepCost{2.6, 0.75, 0.75, 1.7, 0.8, 1.7};
  // clusters do not reach every SM; CTAs beyond one an SM come two at a time where two fit
  const double ctas = (double)g.de * pl.cs, sms = num_sms, reach = pl.cs > 1 ? 0.85 * sms : sms;
  const bool two = pl.smem <= kPlaneSmemGoal;
  const double busiest = ctas <= reach ? 1.0 : std::max(2.0, std::ceil(ctas / (two ? sms : reach)));
  const double waves =
      std::ceil(ctas / ((two && pl.bx * pl.by <= kPlaneThreads / 2 ? 2.0 : 1.0) * reach));
  const double lines = std::min(pl.lines, g.ny) + (pl.cs > 1 ? 1.5 : 0.0);   // with the halo
  const double elements = lines * 2.0 * pl.bx * V / 1000.0 * (vec ? 1.0 : 1.5);
  const double rounds = (pl.lines / 2 + 2 + pl.by - 1) / pl.by;
  const double body = c.work * busiest * elements + c.round * waves * rounds;
  // without odd planes one launch runs seven phases, otherwise three run fifteen
  const double planes = g.dO > 0 ? 3.0 * (c.launch + body) : c.launch + 5.0 / 3.0 * body;
  double phases = 0.0, points = 0.0;
  for (int q = 0; q < kColours; ++q) {
    const double times = q < kColours - 1 ? 2.0 : 1.0;
    if (L.cnt[q] > 0) phases += times;
    points += times * (double)L.cnt[q];
  }
  return std::max(c.least * phases, c.phase * phases + c.element * points * g.R / sms / 1000.0) <
         planes;
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
  bool vec = true;
  const int V = plane_elems(g, r, z, &vec);
  const bool fits = V == 4   ? plane_plan<T, 4>(g, h->num_sms, &pl)
                    : V == 2 ? plane_plan<T, 2>(g, h->num_sms, &pl)
                             : plane_plan<T, 1>(g, h->num_sms, &pl);
  if (!fits || (R > 1 && !vec) || by_colours<T>(g, L, pl, V, vec, h->num_sms)) {
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
                  return from_zero ? plane_launch<T, kOddFwd, true>(h, g, V, vec, pl, r, diag, z, c0_done, s)
                                   : plane_launch<T, kOddFwd, false>(h, g, V, vec, pl, r, diag, z, c0_done, s);
                }, phases(c0_done ? 1 : 0, 3));
    if (rc) return rc;
  }
  rc = launch(h, K_GS, level, prec, (half[1] * 2 + (from_zero ? half[0] : all)) * sv, s,
              "gs_plane_kernel", [&] {
                return from_zero ? plane_launch<T, kEven, true>(h, g, V, vec, pl, r, diag, z, 0, s)
                                 : plane_launch<T, kEven, false>(h, g, V, vec, pl, r, diag, z, 0, s);
              }, phases(4, 7) + phases(4, 6));
  if (rc || g.dO == 0) return rc;
  return launch(h, K_GS, level, prec, (half[0] * 2 + all) * sv, s, "gs_plane_kernel",
                [&] { return plane_launch<T, kOddBwd, false>(h, g, V, vec, pl, r, diag, z, 0, s); },
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
