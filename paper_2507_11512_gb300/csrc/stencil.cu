// Products with the 27-point operator evaluated straight from the grid: SpMV
// and the fused residual-restriction, for one right-hand side and for
// R-vectors.
//
// See stencil.cuh for what they read and why their values equal the ELL
// kernels' bit for bit.

#include <algorithm>

#include "stencil.cuh"

namespace hpg {

// ------------------------------------------------------------------ product
// y = A x (Sec. 3.2.2).  FP32: instruction issue first, then the vectors'
// traffic (8 bytes a row); FP64: the FP64 rate (27 FMAs a row).  A thread takes
// an element group of LINES consecutive x-lines, so that a warp's loads run
// along x, neighbour lines are reused in registers and two FP32 elements share
// loads and addresses.  GB300, stored matrix -> this: FP32 128^3 74 -> 9.1 us, 320^3
// 1.2 ms -> 117 us; FP64 96^3 57 -> 45 us, 128^3 128 -> 99 us.
template <typename T, int R, bool VEC, int LINES>
__global__ void __launch_bounds__(256)
stencil_spmv_kernel(const __grid_constant__ SGeom g, const __grid_constant__ Coef<T> c,
                    const __grid_constant__ RowPlan pl, const T* x, const T* diag, T* y) {
  constexpr int V = row_elems<T>();
  pdl_trigger();
  pdl_wait();
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < pl.threads) {
    const unsigned e = t % pl.across, q = t / pl.across;
    const unsigned grp = q % pl.groups, k = q / pl.groups;
    stencil_rows<T, 1, R, V, VEC, LINES>(
        g, c, x, diag, (int)e * V, (int)grp * LINES, (int)k,
        [](unsigned, const bool (&)[V], T (&a)[V]) {
#pragma unroll
          for (int v = 0; v < V; ++v) a[v] = T(0);
        },
        [&](unsigned p, const bool (&m)[V], const T (&a)[V]) {
          store_elems<T, V, VEC>(y + p, m, a);
        });
  } else if (t - pl.threads < pl.pad) {
    const unsigned p = pad_element(g, t - pl.threads);
    y[p] = ld_dep(x + p);
  }
}

// The same with one thread per storage row, for FP64 levels between these sizes,
// whose FP64 work single rows spread most evenly over the SMs (rows against pairs
// of lines: 40^3 6.2 / 7.0 us, 72^3 20.9 / 23.9, 96^3 44.7 / 45.5; 128^3 101 / 99).
constexpr long long kRowPoints64 = 60000, kRowPointsMax64 = 1500000;
__global__ void __launch_bounds__(64)
stencil_spmv_row_kernel(const __grid_constant__ SGeom g, const __grid_constant__ Coef<double> c,
                        unsigned ns, const double* x, const double* diag, double* y) {
  pdl_trigger();
  const unsigned row = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_wait();
  if (row >= ns) return;
  double v = 0.0;
  const bool point = for_row_slots(g, row, [&](int s, int ci, bool in, unsigned q) {
    const double a = s == kCentre ? (diag ? diag[row] : kDiag) : in ? c.a[ci] : 0.0;
    v = fma(a, ld_dep(x + q), v);
  });
  y[row] = point ? v : ld_dep(x + row);   // padding row: identity
}

// FP64 levels below kRowPoints64: one thread per point, a row of the grid of blocks per
// colour.  Bound by launch and latency, so every load issues at once from addresses
// formed before the wait (16^3 4.1 us by lines, 2.8 here; 36^3 5.6 / 4.9; against the rows
// above 40^3 6.2 / 6.2, 64^3 15.6 / 17.2: the 72 registers leave too few threads an SM).
struct PointGeom {   // across, lines: by parity
  SGeom g;
  Div31 across[2], lines[2];
};
__global__ void __launch_bounds__(64)
stencil_spmv_point_kernel(const __grid_constant__ PointGeom P, const __grid_constant__ Coef<double> c,
                          const double* x, const double* diag, double* y) {
  pdl_trigger();
  const int colour = (int)blockIdx.y;
  const ColourPlan g = make_colour_plan(P.g, colour, P.across[colour_parity_x(colour)],
                                        P.lines[colour_parity_y(colour)]);
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x, row = g.off + t;
  if (row >= g.end) return;
  if (t >= g.cnt) {   // padding row: identity
    pdl_wait();
    y[row] = ld_dep(x + row);
    return;
  }
  const ColourPlace at(g, t, 1);
  const double dg = diag ? diag[row] : kDiag;
  pdl_wait();
  double v[kSlots], acc = 0.0;
#pragma unroll
  for (int s = 0; s < kSlots; ++s) {
    v[s] = 0.0;
    if (at.in(s)) v[s] = ld_dep(x + at.at(g, s));
  }
#pragma unroll
  for (int s = 0; s < kSlots; ++s)
    acc = fma(s == kCentre ? dg : c.a[s % 3 - 1 + (s / 3) % 3 - 1 + s / 9 - 1 + 3], v[s], acc);
  if (at.edge()) pad_slot(v[kCentre], acc);
  y[row] = acc;
}

RowPlan make_row_plan(const SGeom& g, int elems, int lines) {
  RowPlan p;
  p.across = (unsigned)((g.we + elems - 1) / elems);
  p.groups = (unsigned)((g.ny + lines - 1) / lines);
  p.threads = p.across * p.groups * (unsigned)g.nz;
  p.pad = 0;
  for (int c = 0; c < kColours; ++c) p.pad += g.end[c] - g.off[c] - g.cnt[c];
  return p;
}

// lines a thread takes: as many as leave every SM enough threads (FP32 64^3 4.6 us
// with one, 3.3 with two; 96^3 9.9 / 5.8 / 5.4 with one, two, four); FP64 levels come
// here large
template <typename T> static RowPlan spmv_plan(const SGeom& g, int* lines) {
  constexpr int V = row_elems<T>();
  const long long groups = (long long)((g.we + V - 1) / V) * g.ny * g.nz;
  *lines = sizeof(T) == 8 ? 2 : groups < 25000 ? 1 : groups < 150000 ? 2 : kRowLines;
  return make_row_plan(g, V, *lines);
}
// whether the block size is the caller's: small blocks spread few threads over all SMs,
// and FP64 work evenly (an SM has one FP64 unit, 16 cycles a warp instruction)
template <typename T> static bool spmv_takes_block(const hpg_problem* h, const RowPlan& pl) {
  return sizeof(T) == 4 && (long long)pl.threads > 256LL * h->num_sms;
}
bool stencil_spmv_takes_block(const hpg_problem* h, int level, int R) {
  int lines;
  return spmv_takes_block<float>(h, spmv_plan<float>(make_sgeom(h->lev[level].g, R), &lines));
}

template <typename T, int R, bool VEC>
static cudaError_t spmv_launch(hpg_problem* h, const SGeom& g, const T* x, const T* diag, T* y,
                               int block, cudaStream_t s) {
  int lines;
  const RowPlan pl = spmv_plan<T>(g, &lines);
  if (!spmv_takes_block<T>(h, pl)) block = 64;
  auto fn = stencil_spmv_kernel<T, R, VEC, 2>;
  if constexpr (sizeof(T) == 4) {
    if (lines == 1) fn = stencil_spmv_kernel<T, R, VEC, 1>;
    if (lines == kRowLines) fn = stencil_spmv_kernel<T, R, VEC, kRowLines>;
  }
  return kl(h, fn,
            grid_for((long long)pl.threads + pl.pad, block), block, s, g, make_coef<T>(h->beta),
            pl, x, diag, y);
}

static cudaError_t spmv_points(hpg_problem* h, const SGeom& g, const double* x,
                               const double* diag, double* y, cudaStream_t s) {
  PointGeom P;
  P.g = g;
  P.across[0] = Div31((unsigned)g.we);
  P.across[1] = Div31((unsigned)g.wo);
  P.lines[0] = Div31((unsigned)g.he);
  P.lines[1] = Div31((unsigned)g.ho);
  unsigned most = 0;
  for (int c = 0; c < kColours; ++c) most = std::max(most, g.end[c] - g.off[c]);
  return kl(h, stencil_spmv_point_kernel, dim3((unsigned)grid_for(most, 64), kColours), 64, s, P,
            make_coef<double>(h->beta), x, diag, y);
}

template <typename T>
static int spmv_t(hpg_problem* h, int level, int R, const T* x, T* y, cudaStream_t s,
                  int block) {
  const Level& L = h->lev[level];
  const SGeom g = make_sgeom(L.g, R);
  const T* diag = level_diag<T>(L);
  return launch(h, K_SPMV, level, sizeof(T) == 8 ? HPG_FP64 : HPG_FP32,
                (double)L.n * R * 2.0 * sizeof(T) + (diag ? L.n * (double)sizeof(T) : 0.0), s,
                "stencil_spmv_kernel", [&] {
                  if constexpr (sizeof(T) == 8) {
                    if (L.n < kRowPoints64) return spmv_points(h, g, x, diag, y, s);
                    if (L.n < kRowPointsMax64)
                      return kl(h, stencil_spmv_row_kernel, grid_for(L.g.n_store, 64), 64, s, g,
                                make_coef<double>(h->beta), (unsigned)L.g.n_store, x, diag, y);
                  }
                  const bool vec = whole_groups<T, row_elems<T>()>(g, x, y);
                  if constexpr (sizeof(T) == 4) {   // R-vectors are FP32
                    auto fn = R == 8   ? (vec ? spmv_launch<T, 8, true> : spmv_launch<T, 8, false>)
                              : R == 4 ? (vec ? spmv_launch<T, 4, true> : spmv_launch<T, 4, false>)
                              : R == 2 ? (vec ? spmv_launch<T, 2, true> : spmv_launch<T, 2, false>)
                              : vec    ? spmv_launch<T, 1, true> : spmv_launch<T, 1, false>;
                    return fn(h, g, x, diag, y, block, s);
                  }
                  return spmv_launch<T, 1, true>(h, g, x, diag, y, block, s);
                });
}
int stencil_spmv(hpg_problem* h, int level, int R, const float* x, float* y, cudaStream_t s,
                 int block) {
  return spmv_t<float>(h, level, R, x, y, s, block);
}
int stencil_spmv(hpg_problem* h, int level, int R, const double* x, double* y, cudaStream_t s,
                 int block) {
  return spmv_t<double>(h, level, R, x, y, s, block);
}

// -------------------------------------------------------------- restriction
// Fused residual + injection restriction (Sec. 3.2.4): rc_I = r_f - (A z)_f at
// the fine points f = 2I, which are colour block 7 in the coarse grid's own
// order.  One thread per coarse element; slot order as the product's.  Bound by L2
// latency: 128^3 FP32 12-15 us on the stored matrix, about 5 us now.
// zc0 (optional): the coarse level's first phase from zero on its colour-0
// points, z_I = rc_I / a_II (see symgs).
template <typename T>
__device__ __forceinline__ T sub_line(const Coef<T>& c, int dyz, T l, T m, T r, T acc) {
  return fma(-c.a[dyz + 4], r, fma(-c.a[dyz + 3], m, fma(-c.a[dyz + 2], l, acc)));
}

template <typename T>
__global__ void __launch_bounds__(256)
stencil_restrict_kernel(const __grid_constant__ SGeom gf, const __grid_constant__ Geom gc,
                        const __grid_constant__ Coef<T> c, const T* r, const T* z,
                        const T* fdiag, const T* cdiag, T* rc, T* zc0) {
  pdl_trigger();
  pdl_wait();
  const unsigned p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= gf.cnt[kCoarseColour]) return;
  const unsigned e = p % (unsigned)gf.we, q = p / (unsigned)gf.we;
  const int J = (int)(q % (unsigned)gf.he), K = (int)(q / (unsigned)gf.he);
  const unsigned row = gf.off[kCoarseColour] + p;
  const int j = 2 * J, k = 2 * K;
  T l[9], m[9], rr[9];
#pragma unroll
  for (int u = 0; u < 9; ++u) {
    const int jj = j + u % 3 - 1, kk = k + u / 3 - 1;
    l[u] = m[u] = rr[u] = T(0);
    if ((unsigned)jj < (unsigned)gf.ny && (unsigned)kk < (unsigned)gf.nz) {
      const T* od = z + line_base(gf, 1, jj, kk) + e;
      m[u] = ld_dep(z + line_base(gf, 0, jj, kk) + e);
      if ((int)e >= gf.R && (int)e - gf.R < gf.wo) l[u] = ld_dep(od - gf.R);
      if ((int)e < gf.wo) rr[u] = ld_dep(od);
    }
  }
  T acc = ld_dep(r + row);
  const unsigned I = e / (unsigned)gf.R;
  const T d = fdiag ? fdiag[row / (unsigned)gf.R] : (T)kDiag;
#pragma unroll
  for (int u = 0; u < 9; ++u) {
    const int dyz = u % 3 - 1 + u / 3 - 1;
    if (u == 4) {
      acc = fma(-c.a[2], l[u], acc);
      acc = fma(-d, m[u], acc);
      acc = fma(-c.a[4], rr[u], acc);
      if (x_edge(gf, 0, (int)e) || j == 0 || j == gf.ny - 1 || k == 0 || k == gf.nz - 1)
        pad_slot(m[u], acc);
    } else {
      acc = sub_line(c, dyz, l[u], m[u], rr[u], acc);
    }
  }
  const long long Rc = store_index(gc, (int)I, J, K);
  rc[Rc * gf.R + (e - I * gf.R)] = acc;
  if (zc0 && colour_of((int)I, J, K) == 0)
    zc0[Rc * gf.R + (e - I * gf.R)] = acc / (cdiag ? cdiag[Rc] : (T)kDiag);
}

template <typename T>
static int restrict_t(hpg_problem* h, int level, int R, const T* r, const T* z, T* rc, T* zc0,
                      cudaStream_t s) {
  const Level& L = h->lev[level];
  const Level& C = h->lev[level + 1];
  const SGeom g = make_sgeom(L.g, R);
  const double cnt = (double)g.cnt[kCoarseColour];
  // z is read once, r and rc once per coarse row
  return launch(h, K_RESTRICT, level, sizeof(T) == 8 ? HPG_FP64 : HPG_FP32,
                ((double)L.n * R + 2.0 * cnt) * sizeof(T), s, "stencil_restrict_kernel", [&] {
                  return kl(h, stencil_restrict_kernel<T>, grid_for((long long)cnt, 256), 256, s,
                            g, C.g, make_coef<T>(h->beta), r, z, level_diag<T>(L),
                            level_diag<T>(C), rc, zc0);
                });
}
int stencil_restrict(hpg_problem* h, int level, int R, const float* r, const float* z, float* rc,
                     float* zc0, cudaStream_t s) {
  return restrict_t<float>(h, level, R, r, z, rc, zc0, s);
}
int stencil_restrict(hpg_problem* h, int level, int R, const double* r, const double* z,
                     double* rc, double* zc0, cudaStream_t s) {
  return restrict_t<double>(h, level, R, r, z, rc, zc0, s);
}

}  // namespace hpg
