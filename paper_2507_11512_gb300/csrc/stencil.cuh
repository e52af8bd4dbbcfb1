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
// kernels here take R at run time and serve one right-hand side with R = 1;
// the arithmetic of a column does not depend on R.
//
// Values equal those of the ELL kernels bit for bit: same coefficients, same
// order of the products.  A neighbour outside the grid is an ELL padding slot
// there (column = own row, value 0); here it contributes nothing, and one
// product 0 * (own entry) on boundary rows keeps the effect such a slot has
// when the own entry is infinite or NaN.
#pragma once

#include "hpg_internal.cuh"

namespace hpg {

// Slot visited q-th by a Gauss-Seidel phase: the plane below, the plane above,
// then the point's own plane.  Both outer planes have the other z parity and
// are constant while the colours of one plane parity are updated, so their 18
// products are formed once for several updates of a point (gs_plane_kernel).
__host__ __device__ constexpr int gs_order(int q) { return q < 9 ? q : q < 18 ? q + 9 : q - 9; }

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

// What the two points at element e of line (j, k) -- x = 2I and x = 2I + 1 --
// touch on that line: x = 2I-1, 2I, 2I+1, 2I+2.  Zero outside the grid.
template <typename T> struct LinePts { T l, e, o, r; };
template <typename T>
__device__ __forceinline__ LinePts<T> load_line(const T* v, const SGeom& g, int j, int k, int e) {
  LinePts<T> p;
  p.l = p.e = p.o = p.r = T(0);
  if ((unsigned)j < (unsigned)g.ny && (unsigned)k < (unsigned)g.nz) {
    const T* ev = v + line_base(g, 0, j, k) + e;
    const T* od = v + line_base(g, 1, j, k) + e;
    if (e < g.we) p.e = ld_dep(ev);
    if (e < g.wo) p.o = ld_dep(od);
    if (e >= g.R && e - g.R < g.wo) p.l = ld_dep(od - g.R);
    if (e + g.R < g.we) p.r = ld_dep(ev + g.R);
  }
  return p;
}

// acc + sum over the three points dx = -1..1 of a line at offset (dy, dz) of
// a * x, for the even (px = 0) or odd point; sign: +1 adds, -1 subtracts the
// products (fma of the negated coefficient, as the ELL kernels do).
template <typename T, int SIGN>
__device__ __forceinline__ T line_sum(const Coef<T>& c, int dyz, T l, T m, T r, T acc) {
  const T a0 = c.a[dyz + 2], a1 = c.a[dyz + 3], a2 = c.a[dyz + 4];
  acc = fma(SIGN > 0 ? a0 : -a0, l, acc);
  acc = fma(SIGN > 0 ? a1 : -a1, m, acc);
  return fma(SIGN > 0 ? a2 : -a2, r, acc);
}

// Whether a point touches the grid's boundary.
__device__ __forceinline__ bool on_boundary(const SGeom& g, int i, int j, int k) {
  return i == 0 || i == g.nx - 1 || j == 0 || j == g.ny - 1 || k == 0 || k == g.nz - 1;
}

// acc + SIGN * A_ij x_j over all 27 slots in slot order, for the point pair at
// element e of line (j, k); w[dz][dy] are the lines around it.  diag: the
// diagonal entry of each point.
template <typename T, int SIGN, bool ODD>
__device__ __forceinline__ T point_sum(const Coef<T>& c, const LinePts<T> (&w)[3][3], T diag,
                                       bool boundary, T acc) {
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
      const LinePts<T>& p = w[dz + 1][dy + 1];
      const T l = ODD ? p.e : p.l, m = ODD ? p.o : p.e, r = ODD ? p.r : p.o;
      if (dy == 0 && dz == 0) {
        acc = fma(SIGN > 0 ? c.a[2] : -c.a[2], l, acc);
        acc = fma(SIGN > 0 ? diag : -diag, m, acc);
        acc = fma(SIGN > 0 ? c.a[4] : -c.a[4], r, acc);
        if (boundary) acc = fma(T(0), m, acc);
      } else {
        acc = line_sum<T, SIGN>(c, dy + dz, l, m, r, acc);
      }
    }
  return acc;
}

// Lines a thread of a whole-grid product takes (stencil_rows): 4 share their
// neighbour lines in registers (72 loads for 8 rows instead of 144); 1 where
// that would leave SMs without work.
constexpr int kRowLines = 4;

// f(row element, sum, boundary) for every point of up to LINES consecutive
// lines of plane k at element e, where sum = init(element) + SIGN * (A x).
template <typename T, int SIGN, int LINES, typename Init, typename Out>
__device__ __forceinline__ void stencil_rows(const SGeom& g, const Coef<T>& c, const T* x,
                                             const T* diag, int e, int j0, int k, Init&& init,
                                             Out&& out) {
  LinePts<T> w[3][3];
#pragma unroll
  for (int dz = 0; dz < 3; ++dz) {
    w[dz][1] = load_line(x, g, j0 - 1, k + dz - 1, e);
    w[dz][2] = load_line(x, g, j0, k + dz - 1, e);
  }
#pragma unroll
  for (int q = 0; q < LINES; ++q) {
    const int j = j0 + q;
    if (j >= g.ny) break;
#pragma unroll
    for (int dz = 0; dz < 3; ++dz) {
      w[dz][0] = w[dz][1];
      w[dz][1] = w[dz][2];
      w[dz][2] = load_line(x, g, j + 1, k + dz - 1, e);
    }
    const int I2 = e / g.R * 2;
    if (e < g.we) {
      const unsigned p = line_base(g, 0, j, k) + e;
      const T d = diag ? diag[p / (unsigned)g.R] : (T)kDiag;
      out(p, point_sum<T, SIGN, false>(c, w, d, on_boundary(g, I2, j, k), init(p)));
    }
    if (e < g.wo) {
      const unsigned p = line_base(g, 1, j, k) + e;
      const T d = diag ? diag[p / (unsigned)g.R] : (T)kDiag;
      out(p, point_sum<T, SIGN, true>(c, w, d, on_boundary(g, I2 + 1, j, k), init(p)));
    }
  }
}

// Threads of a whole-grid product with LINES lines each: (element, line group,
// plane), plus one thread per padding row element at the end.
struct RowPlan {
  int lines;              // 1 or kRowLines
  unsigned groups;        // line groups per plane
  unsigned threads;       // point threads
  unsigned pad;           // padding elements
};
RowPlan make_row_plan(const SGeom& g, int lines);

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
