// The 27-point operator applied straight from its grid (no stored matrix):
// geometry, coefficients and the neighbour loads shared by the kernels that
// evaluate it (stencil.cu, krylov.cu).
//
// An off-diagonal entry depends only on s = dx + dy + dz (-1 + beta s / 3, Sec.
// 3) and a neighbour's storage row only on the grid position, so a product or
// a Gauss-Seidel phase needs neither the 27 values nor the 27 column indices
// of a row: of the 224 bytes a row of the FP32 ELL form costs, the 8 to 12
// bytes of its vector entries remain.  The ELL arrays stay for the
// implementation options that run on them.
//
// An R-vector ([n_store][R], R right-hand sides of one problem) is the same
// thing with every line R times as wide and a step in x of R elements, so all
// kernels here serve one right-hand side with R = 1; the arithmetic of a column
// does not depend on R.
//
// Values equal those of the ELL kernels bit for bit: same coefficients, same
// order of the products (pad_slot covers neighbours outside the grid).
#pragma once

#include "hpg_internal.cuh"

namespace hpg {

// A level's geometry in elements of an R-vector.  e / o: even / odd
// coordinate.  off32 holds fewer than 2^31 elements (n_store * 27 < 2^31).
struct SGeom {
  int nx, ny, nz, R;
  int we, wo;        // elements of the even / odd part of an x-line
  int he, ho;        // lines of the even / odd y parity in a plane
  int de, dO;        // planes of the even / odd z parity
  unsigned off[kColours], cnt[kColours], end[kColours];   // blocks (end: with padding)
};

inline SGeom make_sgeom(const Geom& g, int R) {
  SGeom s;
  s.nx = g.nx; s.ny = g.ny; s.nz = g.nz; s.R = R;
  s.we = (g.nx + 1) / 2 * R; s.wo = g.nx / 2 * R;
  s.he = (g.ny + 1) / 2; s.ho = g.ny / 2;
  s.de = (g.nz + 1) / 2; s.dO = g.nz / 2;
  for (int c = 0; c < kColours; ++c) {
    s.off[c] = (unsigned)(g.off[c] * R);
    s.cnt[c] = (unsigned)((long long)g.cdx[c] * g.cdy[c] * g.cdz[c] * R);
    s.end[c] = (unsigned)(g.off[c + 1] * R);
  }
  return s;
}

// Off-diagonal entries by s + 3, in the working precision (the values
// gen_ell_kernel writes).
template <typename T> struct Coef { T a[7]; };
template <typename T> inline Coef<T> make_coef(double beta) {
  Coef<T> c;
  for (int s = -3; s <= 3; ++s) c.a[s + 3] = (T)(-1.0 + beta * (double)s / 3.0);
  return c;
}

// First element of the x-line (j, k), x parity px (0 even, 1 odd).
__device__ __forceinline__ unsigned line_base(const SGeom& g, int px, int j, int k) {
  const int c = (px ^ 1) | (((j & 1) ^ 1) << 1) | (((k & 1) ^ 1) << 2);
  const int w = px ? g.wo : g.we, h = (j & 1) ? g.ho : g.he;
  return g.off[c] + (unsigned)w * ((unsigned)(j >> 1) + (unsigned)h * (unsigned)(k >> 1));
}

// A thread takes V consecutive elements of an x-line, each standing for the
// two points x = 2I and x = 2I + 1.  LinePts holds what they touch on one line:
// x = 2I-1 (l), 2I (e), 2I+1 (o), 2I+2 (r), zero outside the grid.
template <typename T, int V> struct LinePts { T l[V], e[V], o[V], r[V]; };

// Which of a thread's elements exist (they depend on its position in x only).
// VEC: the elements of a part come in whole, aligned groups of V.
template <int R, int V, bool VEC> struct XMask {
  bool e[V], o[V], l[V], r[V];
  __device__ __forceinline__ XMask(const SGeom& g, int x) {
#pragma unroll
    for (int v = 0; v < V; ++v) {
      e[v] = VEC ? x < g.we : x + v < g.we;
      o[v] = VEC ? x < g.wo : x + v < g.wo;
      l[v] = x + v >= R && x + v - R < g.wo;
      r[v] = x + v + R < g.we;
    }
  }
};

template <typename T, int V> struct VecOf { using type = T; };
template <> struct VecOf<float, 2> { using type = float2; };
template <> struct VecOf<float, 4> { using type = float4; };
__device__ __forceinline__ void unpack(float v, float (&o)[1]) { o[0] = v; }
__device__ __forceinline__ void unpack(double v, double (&o)[1]) { o[0] = v; }
__device__ __forceinline__ void unpack(float2 v, float (&o)[2]) { o[0] = v.x; o[1] = v.y; }
__device__ __forceinline__ void unpack(float4 v, float (&o)[4]) {
  o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}

// The line whose even and odd parts start (at the thread's element) at ev, od;
// in: the line exists.
template <typename T, int R, int V, bool VEC>
__device__ __forceinline__ LinePts<T, V> load_line(const T* ev, const T* od, bool in,
                                                   const XMask<R, V, VEC>& m) {
  LinePts<T, V> p;
#pragma unroll
  for (int v = 0; v < V; ++v) p.l[v] = p.e[v] = p.o[v] = p.r[v] = T(0);
  if (!in) return p;
  if constexpr (VEC && V > 1) {
    using P = typename VecOf<T, V>::type;
    unpack(ld_dep(reinterpret_cast<const P*>(ev)), p.e);
    if (m.o[0]) unpack(ld_dep(reinterpret_cast<const P*>(od)), p.o);
    if constexpr (R % V == 0) {
      if (m.l[0]) unpack(ld_dep(reinterpret_cast<const P*>(od - R)), p.l);
      if (m.r[0]) unpack(ld_dep(reinterpret_cast<const P*>(ev + R)), p.r);
    } else {   // R = 1
      if (m.l[0]) p.l[0] = ld_dep(od - 1);
      if (m.r[V - 1]) p.r[V - 1] = ld_dep(ev + V);
#pragma unroll
      for (int v = 1; v < V; ++v) {
        p.l[v] = p.o[v - 1];
        p.r[v - 1] = p.e[v];
      }
    }
  } else {
#pragma unroll
    for (int v = 0; v < V; ++v) {
      if (m.e[v]) p.e[v] = ld_dep(ev + v);
      if (m.o[v]) p.o[v] = ld_dep(od + v);
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
      if (V > R && v >= R) p.l[v] = p.o[v - R];
      else if (m.l[v]) p.l[v] = ld_dep(od + v - R);
      if (V > R && v + R < V) p.r[v] = p.e[v + R];
      else if (m.r[v]) p.r[v] = ld_dep(ev + v + R);
    }
  }
  return p;
}

// Start of a plane's lines at element x: line j (parity p = j & 1) begins at
// ev[p] + (j >> 1) * we and od[p] + (j >> 1) * wo.
template <typename T> struct PlanePtr {
  const T *ev[2], *od[2];
  __device__ __forceinline__ PlanePtr(const T* v, const SGeom& g, int k, int x) {
    const int K = k >> 1, cz = (k & 1) ? 0 : 4;
    ev[0] = v + (g.off[cz | 3] + (unsigned)g.we * (unsigned)(g.he * K) + x);
    od[0] = v + (g.off[cz | 2] + (unsigned)g.wo * (unsigned)(g.he * K) + x);
    ev[1] = v + (g.off[cz | 1] + (unsigned)g.we * (unsigned)(g.ho * K) + x);
    od[1] = v + (g.off[cz] + (unsigned)g.wo * (unsigned)(g.ho * K) + x);
  }
};

// acc + the products of one line at dy + dz = dyz, for the even and odd points;
// SIGN -1 subtracts them (fma of the negated coefficient, as the ELL kernels).
template <typename T, int SIGN, int V>
__device__ __forceinline__ void line_sum(const Coef<T>& c, int dyz, const LinePts<T, V>& p,
                                         T (&ae)[V], T (&ao)[V]) {
  const T a0 = SIGN > 0 ? c.a[dyz + 2] : -c.a[dyz + 2];
  const T a1 = SIGN > 0 ? c.a[dyz + 3] : -c.a[dyz + 3];
  const T a2 = SIGN > 0 ? c.a[dyz + 4] : -c.a[dyz + 4];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    ae[v] = fma(a2, p.o[v], fma(a1, p.e[v], fma(a0, p.l[v], ae[v])));
    ao[v] = fma(a2, p.r[v], fma(a1, p.o[v], fma(a0, p.e[v], ao[v])));
  }
}

// The same for one point of parity XO of element v.
template <typename T, bool XO, int V>
__device__ __forceinline__ T half_sum(const Coef<T>& c, int dyz, const LinePts<T, V>& p, int v,
                                      T acc) {
  const T l = XO ? p.e[v] : p.l[v], q = XO ? p.o[v] : p.e[v], r = XO ? p.r[v] : p.o[v];
  return fma(-c.a[dyz + 4], r, fma(-c.a[dyz + 3], q, fma(-c.a[dyz + 2], l, acc)));
}

// x / 26, correctly rounded: Markstein's division by a known divisor (IBM J.
// Res. Dev. 34, 1990): with y = RN(1/26), q = RN(x y) and the exact remainder
// x - 26 q, RN(q + remainder * y) is RN(x / 26) unless something under- or
// overflows, which the range test leaves to the plain division.
__device__ __forceinline__ bool div_safe(float x) {   // 2^-95 <= |x| < 2^123
  return (__float_as_uint(x) & 0x7fffffffu) - 0x10000000u < 0x7d000000u - 0x10000000u;
}
__device__ __forceinline__ bool div_safe(double x) {  // 2^-823 <= |x| < 2^877
  return ((unsigned)__double2hiint(x) & 0x7fffffffu) - (200u << 20) < (1700u << 20);
}
__device__ __forceinline__ float div_known(float x) {
  constexpr float y = 1.0f / (float)kDiag;
  const float q = x * y;
  return fmaf(fmaf(-(float)kDiag, q, x), y, q);
}
__device__ __forceinline__ double div_known(double x) {
  constexpr double y = 1.0 / kDiag;
  const double q = x * y;
  return fma(fma(-kDiag, q, x), y, q);
}
// Out of line: inlined, part of the division runs on the safe path as well
// (FP64 sweeps 20 % slower).
static __device__ __noinline__ float div_plain(float x) { return x / (float)kDiag; }
static __device__ __noinline__ double div_plain(double x) { return x / kDiag; }
template <typename T, int V> __device__ __forceinline__ void div_diag(T (&x)[V]) {
  bool safe = true;
  T q[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    safe = safe && div_safe(x[v]);
    q[v] = div_known(x[v]);
  }
  if (!safe) {
#pragma unroll
    for (int v = 0; v < V; ++v) q[v] = div_plain(x[v]);
  }
#pragma unroll
  for (int v = 0; v < V; ++v) x[v] = q[v];
}

// What an ELL padding slot (own column, value 0) adds on boundary rows: nothing,
// unless the own entry is infinite or NaN.  The test is on its exponent, so that
// FP64 rows do not pay for a product.
__device__ __forceinline__ void pad_slot(float own, float& acc) {
  if ((__float_as_uint(own) & 0x7f800000u) == 0x7f800000u) acc = fmaf(0.0f, own, acc);
}
__device__ __forceinline__ void pad_slot(double own, double& acc) {
  if ((__double2hiint(own) & 0x7ff00000) == 0x7ff00000) acc = fma(0.0, own, acc);
}

// Whether element e of an x-line's even (px 0) or odd part is its first or
// last grid point.
__device__ __forceinline__ bool x_edge(const SGeom& g, int px, int e) {
  return (px == 0 && e < g.R) || (px == ((g.nx - 1) & 1) && e >= (px ? g.wo : g.we) - g.R);
}

// f(slot, coefficient index, inside the grid, neighbour's row or else own row)
// for the 27 slots of a storage row (geometry with R = 1) in slot order; false
// for a padding row.  For kernels with one thread per storage row.
template <typename F>
__device__ __forceinline__ bool for_row_slots(const SGeom& g, unsigned row, F&& f) {
  int colour = 0;
#pragma unroll
  for (int q = 1; q < kColours; ++q) colour += row >= g.off[q] ? 1 : 0;
  const unsigned p = row - g.off[colour];
  if (p >= g.cnt[colour]) return false;
  const int px = colour_parity_x(colour), py = colour_parity_y(colour),
            pz = colour_parity_z(colour);
  const unsigned w = px ? g.wo : g.we, hl = py ? g.ho : g.he;
  const int e = (int)(p % w), i = 2 * e + px;
  const int j = 2 * (int)(p / w % hl) + py, k = 2 * (int)(p / w / hl) + pz;
#pragma unroll
  for (int s = 0; s < kSlots; ++s) {
    const int dx = s % 3 - 1, dy = (s / 3) % 3 - 1, dz = s / 9 - 1;
    const bool in = (unsigned)(i + dx) < (unsigned)g.nx && (unsigned)(j + dy) < (unsigned)g.ny &&
                    (unsigned)(k + dz) < (unsigned)g.nz;
    f(s, dx + dy + dz + 3, in,
      in ? line_base(g, px ^ (dx & 1), j + dy, k + dz) + e + ((px + dx) >> 1) : row);
  }
  return true;
}

// Quotients by a fixed divisor below 2^31 of dividends below 2^31 (Granlund and
// Montgomery, PLDI 1994: the multiplier for 31-bit operands fits 32 bits).
struct Div31 {
  unsigned d, m, sh;
  Div31() = default;
  __host__ explicit Div31(unsigned n) : d(n), m(0), sh(0) {
    if (n <= 1) return;
    sh = 31 - (unsigned)__builtin_clz(n - 1);   // 2^sh < n <= 2^(sh + 1)
    m = (unsigned)((1ULL << (32 + sh)) / n + 1);
  }
  __device__ __forceinline__ unsigned div(unsigned t) const { return m ? __umulhi(t, m) >> sh : t; }
};

// What a kernel with one thread per point of a colour needs of its level, in
// elements of an R-vector.  A
// neighbour's line part is told by which of its parities differ from the colour's:
// flip f (bit 0 x, 1 y, 2 z) starts at o[f] and steps w[f] a line, wh[f] a plane; slot
// s adds d[s].
struct ColourPlan {
  unsigned off, cnt, end;     // the colour's block (end: with padding rows)
  Div31 across, lines;        // a line's element groups, a plane's lines
  int px, py, pz, ny, nz, R, rshift;
  int early;                  // whether the next kernel may start while this one runs
  unsigned o[8], w[8], wh[8];
  int d[kSlots];
};
// across, lines: of the colour's x and y parity.
__host__ __device__ inline ColourPlan make_colour_plan(const SGeom& g, int colour, Div31 across,
                                                      Div31 lines) {
  const int px = colour_parity_x(colour), py = colour_parity_y(colour),
            pz = colour_parity_z(colour);
  ColourPlan q{g.off[colour], g.cnt[colour], g.end[colour], across, lines};
  q.px = px; q.py = py; q.pz = pz; q.ny = g.ny; q.nz = g.nz; q.R = g.R;
  q.rshift = g.R == 8 ? 3 : g.R >> 1;
  q.early = 1;
#pragma unroll
  for (int f = 0; f < 8; ++f) {
    const int x = px ^ (f & 1), y = py ^ (f >> 1 & 1), z = pz ^ (f >> 2);
    q.o[f] = g.off[(x ^ 1) | (y ^ 1) << 1 | (z ^ 1) << 2];
    q.w[f] = (unsigned)(x ? g.wo : g.we);
    q.wh[f] = q.w[f] * (unsigned)(y ? g.ho : g.he);
  }
#pragma unroll
  for (int s = 0; s < kSlots; ++s) {
    const int dx = s % 3 - 1, dy = (s / 3) % 3 - 1, dz = s / 9 - 1;
    const int f = (dx & 1) | (dy & 1) << 1;   // w and wh do not depend on the z parity
    q.d[s] = ((px + dx) >> 1) * g.R + ((py + dy) >> 1) * (int)q.w[f] +
             ((pz + dz) >> 1) * (int)q.wh[f];
  }
  return q;
}

// A thread's place in a colour (element p = V t of its block): line element e, line J
// and plane K of the colour, whether the points before and after exist along x, y
// and z, and the first element of each flip's line part at its place.
struct ColourPlace {
  bool lo[3], up[3];
  unsigned base[8];
  __device__ __forceinline__ ColourPlace(const ColourPlan& g, unsigned t, int V) {
    const unsigned q = g.across.div(t), e = (t - q * g.across.d) * V;
    const unsigned K = g.lines.div(q), J = q - K * g.lines.d;
    const int j = 2 * (int)J + g.py, k = 2 * (int)K + g.pz;
    lo[0] = g.px || e >= (unsigned)g.R;
    up[0] = e + (unsigned)(g.px * g.R) < g.w[1];
    lo[1] = j > 0, up[1] = j + 1 < g.ny;
    lo[2] = k > 0, up[2] = k + 1 < g.nz;
#pragma unroll
    for (int f = 0; f < 8; ++f) {
      base[f] = g.o[f] + g.w[f] * J + g.wh[f] * K + e;
      asm volatile("" : "+r"(base[f]));   // formed here, not after the caller's wait
    }
  }
  __device__ __forceinline__ bool edge() const {
    return !(lo[0] && up[0] && lo[1] && up[1] && lo[2] && up[2]);
  }
  // neighbour at slot s: whether it exists, and its element
  __device__ __forceinline__ bool in(int s) const {
    const int d[3] = {s % 3 - 1, (s / 3) % 3 - 1, s / 9 - 1};
    bool v = true;
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (d[a]) v = v && (d[a] < 0 ? lo[a] : up[a]);
    return v;
  }
  __device__ __forceinline__ unsigned at(const ColourPlan& g, int s) const {
    const int dx = s % 3 - 1, dy = (s / 3) % 3 - 1, dz = s / 9 - 1;
    return base[(dx & 1) | (dy & 1) << 1 | (dz & 1) << 2] + (unsigned)g.d[s];
  }
};

// Lines a thread of a whole-grid product takes (stencil_rows), at most: they
// share their neighbour lines in registers.
constexpr int kRowLines = 4;
// Elements of a line it takes: the loads of two FP32 elements are one load
// each, and their addresses one computation; FP64 is bound by its FMAs.
template <typename T> __host__ __device__ constexpr int row_elems() {
  return sizeof(T) == 4 ? 2 : 1;
}
// Whether a vector's parts come in whole aligned groups of V elements.
template <typename T, int V> inline bool whole_groups(const SGeom& g, const void* a, const void* b) {
  return V == 1 || (g.we % V == 0 && g.wo % V == 0 &&
                    (((uintptr_t)a | (uintptr_t)b) & (V * sizeof(T) - 1)) == 0);
}

// out(first element, V sums, which exist) for the even and the odd points of up
// to LINES lines of plane k from j0 on at element x, with sum = init(first
// element) + SIGN * (A x) over all 27 slots in slot order.
template <typename T, int SIGN, int R, int V, bool VEC, int LINES, typename Init, typename Out>
__device__ __forceinline__ void stencil_rows(const SGeom& g, const Coef<T>& c, const T* xv,
                                             const T* diag, int x, int j0, int k, Init&& init,
                                             Out&& out) {
  const XMask<R, V, VEC> m(g, x);
  const bool in_k[3] = {k > 0, true, k + 1 < g.nz};
  const PlanePtr<T> pp[3] = {PlanePtr<T>(xv, g, in_k[0] ? k - 1 : k, x), PlanePtr<T>(xv, g, k, x),
                             PlanePtr<T>(xv, g, in_k[2] ? k + 1 : k, x)};
  LinePts<T, V> w[3][3];
  auto fetch = [&](int dz, int j) {
    const int p = j & 1, J = j >> 1;
    return load_line<T, R, V, VEC>(pp[dz].ev[p] + J * g.we, pp[dz].od[p] + J * g.wo,
                                   in_k[dz] && j >= 0 && j < g.ny, m);
  };
#pragma unroll
  for (int dz = 0; dz < 3; ++dz) {
    w[dz][1] = fetch(dz, j0 - 1);
    w[dz][2] = fetch(dz, j0);
  }
  bool be[V], bo[V], bx = false;   // points on the grid's x faces
#pragma unroll
  for (int v = 0; v < V; ++v) {
    be[v] = x_edge(g, 0, x + v);
    bo[v] = x_edge(g, 1, x + v);
    bx = bx || be[v] || bo[v];
  }
#pragma unroll
  for (int q = 0; q < LINES; ++q) {
    const int j = j0 + q;
    if (j >= g.ny) break;
#pragma unroll
    for (int dz = 0; dz < 3; ++dz) {
      w[dz][0] = w[dz][1];
      w[dz][1] = w[dz][2];
      w[dz][2] = fetch(dz, j + 1);
    }
    const unsigned pe = line_base(g, 0, j, k) + x, po = line_base(g, 1, j, k) + x;
    T ae[V], ao[V];
    init(pe, m.e, ae);
    init(po, m.o, ao);
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy) {
        const LinePts<T, V>& p = w[dz + 1][dy + 1];
        if (dy != 0 || dz != 0) {
          line_sum<T, SIGN, V>(c, dy + dz, p, ae, ao);
          continue;
        }
        const T a0 = SIGN > 0 ? c.a[2] : -c.a[2], a2 = SIGN > 0 ? c.a[4] : -c.a[4];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          T de = (T)kDiag, dd = (T)kDiag;
          if (diag) {
            if (m.e[v]) de = diag[(pe + v) / R];
            if (m.o[v]) dd = diag[(po + v) / R];
          }
          if (SIGN < 0) de = -de, dd = -dd;
          ae[v] = fma(a2, p.o[v], fma(de, p.e[v], fma(a0, p.l[v], ae[v])));
          ao[v] = fma(a2, p.r[v], fma(dd, p.o[v], fma(a0, p.e[v], ao[v])));
        }
        if (bx || j == 0 || j == g.ny - 1 || k == 0 || k == g.nz - 1) {
          const bool edge = j == 0 || j == g.ny - 1 || k == 0 || k == g.nz - 1;
#pragma unroll
          for (int v = 0; v < V; ++v) {
            if (edge || be[v]) pad_slot(p.e[v], ae[v]);
            if (edge || bo[v]) pad_slot(p.o[v], ao[v]);
          }
        }
      }
    out(pe, m.e, ae);
    out(po, m.o, ao);
  }
}

// V elements of a vector at p (those in m), to and from registers.
template <typename T, int V, bool VEC>
__device__ __forceinline__ void load_elems(const T* p, const bool (&m)[V], T (&a)[V]) {
  if constexpr (VEC && V > 1) {
    if (m[0]) unpack(ld_dep(reinterpret_cast<const typename VecOf<T, V>::type*>(p)), a);
  } else {
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (m[v]) a[v] = ld_dep(p + v);
  }
}
template <typename T, int V, bool VEC>
__device__ __forceinline__ void store_elems(T* p, const bool (&m)[V], const T (&a)[V]) {
  if constexpr (VEC && V == 2) {
    if (m[0]) *reinterpret_cast<float2*>(p) = make_float2(a[0], a[1]);
  } else if constexpr (VEC && V == 4) {
    if (m[0]) *reinterpret_cast<float4*>(p) = make_float4(a[0], a[1], a[2], a[3]);
  } else {
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (m[v]) p[v] = a[v];
  }
}

// Threads of a whole-grid product: (element group, line group, plane), plus one
// thread per padding row element at the end.
struct RowPlan {
  unsigned across;        // element groups of a line
  unsigned groups;        // line groups per plane
  unsigned threads;       // point threads
  unsigned pad;           // padding elements
};
RowPlan make_row_plan(const SGeom& g, int elems, int lines);

// Padding element number q of an R-vector, or the first element past the end.
__device__ __forceinline__ unsigned pad_element(const SGeom& g, unsigned q) {
#pragma unroll
  for (int c = 0; c < kColours; ++c) {
    const unsigned lo = g.off[c] + g.cnt[c], n = g.end[c] - lo;
    if (q < n) return lo + q;
    q -= n;
  }
  return 0xffffffffu;
}

// The diagonal entries a level's kernels read per row: null where all are 26.
template <typename T> inline const T* level_diag(const Level& L);
template <> inline const float* level_diag<float>(const Level& L) {
  return L.theta ? L.v32 + kCentre * L.g.n_store : nullptr;
}
template <> inline const double* level_diag<double>(const Level& L) {
  return L.theta ? L.v64 + kCentre * L.g.n_store : nullptr;
}

// y = A x and rc = restriction of r - A z from `level` to the next (zc0: also
// the coarse level's colour-0 phase from zero, or null), on R-vectors.
int stencil_spmv(hpg_problem* h, int level, int R, const float* x, float* y, cudaStream_t s,
                 int block = 256);
int stencil_spmv(hpg_problem* h, int level, int R, const double* x, double* y, cudaStream_t s,
                 int block = 256);
// Whether an FP32 product of R vectors runs with the given block size.
bool stencil_spmv_takes_block(const hpg_problem* h, int level, int R);
int stencil_restrict(hpg_problem* h, int level, int R, const float* r, const float* z, float* rc,
                     float* zc0, cudaStream_t s);
int stencil_restrict(hpg_problem* h, int level, int R, const double* r, const double* z,
                     double* rc, double* zc0, cudaStream_t s);

// One symmetric sweep (colours 0..7 then 7..0) and one colour phase, in place.
// from_zero: z enters as 0 and is not read.  c0_done: colour 0's first phase
// is already in z.
int stencil_symgs(hpg_problem* h, int level, int R, const float* r, float* z, bool from_zero,
                  bool c0_done, cudaStream_t s);
int stencil_symgs(hpg_problem* h, int level, int R, const double* r, double* z, bool from_zero,
                  bool c0_done, cudaStream_t s);
int stencil_colour_phase(hpg_problem* h, int level, int R, int colour, bool from_zero,
                         const float* r, float* z, cudaStream_t s);
int stencil_colour_phase(hpg_problem* h, int level, int R, int colour, bool from_zero,
                         const double* r, double* z, cudaStream_t s);

}  // namespace hpg
