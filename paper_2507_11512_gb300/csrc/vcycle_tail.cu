// The small levels of a V-cycle in one kernel: every vector of every level from
// the first that fits down to the coarsest lives in the shared memory of one
// thread-block cluster.
//
// Launched one by one, a small level's sweep is three kernels of 4-6 us each,
// nearly all of it launch, instruction-fetch and memory latency (a 16^3 FP64
// V-cycle took 25 launches and 196 us).  Here the V-cycle is a list of
// operations (a stage of a sweep, a restriction, a prolongation) that one loop
// runs, so the code is fetched once; planes are dealt out in z, a plane's
// colour phases need only the CTA's own shared memory, the planes above and
// below come over distributed shared memory, and a cluster barrier ends each
// operation.  Coarse plane K belongs to the CTA of fine plane 2K, so transfers
// between levels stay inside a CTA.
//
// Values are those of gs_plane_kernel, stencil_restrict_kernel and
// prolong_kernel bit for bit (same products in the same order).  The products
// with the plane below are formed once per stage; the plane above comes last in
// slot order, so its lines are read in every phase.

#include <algorithm>

#include "stencil.cuh"

namespace hpg {

constexpr int kTailThreads = 512;
// CTAs of the cluster: 16 (beyond the portable size) where the device can place
// one, else 8.  Measured, V-cycles: 32^3 FP32 77 -> 67 us, 128^3 137 -> 131 us.
constexpr int kTailCtas = 16, kTailPortableCtas = 8;
constexpr int kTailOps = 160;
constexpr size_t kTailSmem = 227u << 10;
// Largest first level, by the points (times right-hand sides) of a CTA: a level of few
// planes has few CTAs, so its total says nothing.  Measured, V-cycles, with the
// level in the cluster / launched by itself: FP32 32^3 (2048 points a CTA) 66 / 71 us,
// 28^3 x 2 (3136) 58 / 62, 40 x 40 x 8 (3200) 70 / 66, 32^3 x 2 (4096) 78 / 72, 64 x 64 x 8
// (8192) 105 / 70, 90 x 88 x 4 (15840) 120 / 64; FP64 16^3 (512) 133 / 146, 20^3 (800)
// 109 / 118, 16 x 16 x 64 (1024) 147 / 145, 24^3 (1152) 158 / 152 (a few SMs' FP64 units
// against all).
constexpr long long kTailPoints32 = 3200, kTailPoints64 = 900;
// A sweep alone pays for one launch instead of three, but loads and stores the level.
// Host and device time of a call, here / by planes: FP32 12^3 (288 points a CTA) 16 /
// 14 us, 16^3 (512) 14 / 14, 33 x 17 x 24 (1122) 17 / 18, 24^3 (1152) 16 / 14, 64 x 64 x 4
// (8192) 35 / 14; FP64 16^3 25 / 27, 24 x 16 x 12 (768) 27 / 27, 24 x 24 x 8 (1152) 34 / 27.
constexpr long long kTailSweepPoints32 = 1140, kTailSweepPoints64 = 600;

// Quotients by a fixed divisor (below 2^16, dividends likewise).
struct FastDiv {
  unsigned d, m;
  __host__ explicit FastDiv(int n = 1) : d((unsigned)std::max(n, 1)) {
    m = d == 1 ? 0u : 0xffffffffu / d + 1u;
  }
  __device__ __forceinline__ unsigned div(unsigned t) const { return m ? __umulhi(t, m) : t; }
};

enum TailOpKind { kTailStage = 0, kTailRestrict = 1, kTailProlong = 2 };
struct TailOp {
  unsigned char kind, level;
  unsigned char parity;   // stage: plane parity
  unsigned char first;    // stage: first of a sweep from zero (no outer products)
  unsigned short steps;   // stage: 2 bits a colour phase, first phase lowest: y odd, x odd
  unsigned char nsteps;
  unsigned char cluster;  // other CTAs read what it wrote (or wrote what is read next)
};

template <typename T> struct TailLevel {
  SGeom g;
  FastDiv we, ny, he;
  int pitch, odd, plane;     // z: line pitch, first odd element, elements of a plane
  int z, r, d;               // shared-memory offsets (elements)
  const T* diag;
};

template <typename T> struct TailParams {
  int nlev, nops, ctas, threads;
  int ppc;                     // planes per CTA on the first level
  int given;                   // z enters as given (sweeps), not as 0
  int sp, elems;               // offset of the sums up to the plane below; elements in all
  Coef<T> c;
  const T* r;
  T* z;
  TailLevel<T> lev[kMaxLevels];
  TailOp op[kTailOps];
};

__device__ __forceinline__ void tail_barrier() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of this CTA's shared-memory object p in CTA `rank` (generic).
template <typename T> __device__ __forceinline__ const T* remote(const T* p, int rank) {
  unsigned long long a;
  asm("mapa.u64 %0, %1, %2;" : "=l"(a) : "l"(p), "r"(rank));
  return reinterpret_cast<const T*>(a);
}

template <typename T>
__device__ __forceinline__ T tail_line(const Coef<T>& c, int dyz, T l, T m, T r, T acc) {
  return fma(-c.a[dyz + 4], r, fma(-c.a[dyz + 3], m, fma(-c.a[dyz + 2], l, acc)));
}

// x / 26 as gs_plane_kernel divides, or by the cell's diagonal.
template <typename T>
__global__ void __launch_bounds__(kTailThreads, 1)
vcycle_tail_kernel(const __grid_constant__ TailParams<T> P) {
  extern __shared__ __align__(16) unsigned char tail_smem[];
  T* sm = reinterpret_cast<T*>(tail_smem);
  const int tid = threadIdx.x;
  unsigned rank;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  pdl_trigger();
  for (int i = tid; i < (P.elems * (int)sizeof(T) + 15) / 16; i += blockDim.x)
    reinterpret_cast<float4*>(tail_smem)[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  __syncthreads();
  // first plane of this CTA on level l, and of the next CTA
  auto first_plane = [&](int l, int c) { return ((c * P.ppc) + (1 << l) - 1) >> l; };
  // diagonals of every level, and the first level's right-hand side
  pdl_wait();
  for (int l = 0; l < P.nlev; ++l) {
    const TailLevel<T>& L = P.lev[l];
    if (l > 0 && !L.diag) continue;
    const int f = first_plane(l, rank), e = min(first_plane(l, rank + 1), L.g.nz);
    const int row = L.g.we + L.g.wo;
    for (unsigned t = tid; t < (unsigned)((e - f) * L.g.ny * L.g.we); t += blockDim.x) {
      const unsigned q = L.we.div(t), x = t - q * L.we.d;
      const unsigned ip = L.ny.div(q), j = q - ip * L.ny.d;
      const unsigned pe = line_base(L.g, 0, j, f + ip) + x, po = line_base(L.g, 1, j, f + ip) + x;
      const bool has_o = (int)x < L.g.wo;
      if (l == 0) {
        sm[L.r + q * row + x] = ld_dep(P.r + pe);
        if (has_o) sm[L.r + q * row + L.g.we + x] = ld_dep(P.r + po);
        if (P.given) {
          T* ln = sm + L.z + ip * L.plane + (j + 1) * L.pitch + x;
          ln[L.g.R] = ld_dep(P.z + pe);
          if (has_o) ln[L.odd] = ld_dep(P.z + po);
        }
      }
      if (L.diag) {
        sm[L.d + q * row + x] = L.diag[pe / (unsigned)L.g.R];
        if (has_o) sm[L.d + q * row + L.g.we + x] = L.diag[po / (unsigned)L.g.R];
      }
    }
  }
  tail_barrier();

  for (int o = 0; o < P.nops; ++o) {
    const TailOp op = P.op[o];
    const TailLevel<T>& L = P.lev[op.level];
    const SGeom& g = L.g;
    const int R = g.R, row = g.we + g.wo;
    const int f = first_plane(op.level, rank);
    const int fe = min(first_plane(op.level, rank + 1), g.nz);
    T* z = sm + L.z;
    const T* r = sm + L.r;
    // plane k of this level's z, wherever it lives
    auto plane_of = [&](int k) -> const T* {
      if (k >= f && k < fe) return z + (k - f) * L.plane;
      const int c = (k << op.level) / P.ppc;
      return remote(z + (k - first_plane(op.level, c)) * L.plane, c);
    };
    if (op.kind == kTailStage) {
      const int k0 = f + ((f ^ op.parity) & 1);
      const int np = fe > k0 ? (fe - k0 + 1) >> 1 : 0;
      const int pitch = L.pitch, odd = L.odd, plane = L.plane, ny = g.ny, we = g.we, wo = g.wo;
      const FastDiv dwe = L.we, dhe = L.he;
      const bool first = op.first;
      const T* diag = L.diag ? sm + L.d : nullptr;
      T* sp = sm + P.sp;
      // the plane above the last own one, if that has this parity, lives in the
      // next CTA: a copy of it
      if (!first && np > 0 && k0 + 2 * (np - 1) + 1 == fe && fe < g.nz) {
        const T* src = plane_of(fe);
        T* dst = z + (fe - f) * plane;
        for (int t = tid; t < plane; t += blockDim.x) dst[t] = src[t];
      }
      // A thread's item: the 2 x 2 points (y even / odd, x even / odd) at (J, x) of
      // a plane, one of each colour, so every phase keeps every thread busy.
      const int items = np * g.he * we;
      T* zb = z;          // the (even, even) point
      int x = 0, j = 0, k = 0, pi = 0;
      unsigned has = 0, bnd = 0;   // bit 2 * yo + xo: the point exists / is a boundary point
      auto locate = [&](int t) {
        const unsigned q = dwe.div(t), ip = dhe.div(q);
        x = t - (int)(q * dwe.d);
        j = 2 * (int)(q - ip * dhe.d);
        k = k0 + 2 * (int)ip;
        pi = ((k - f) * ny + j) * row + x;
        zb = z + (k - f) * plane + (j + 1) * pitch + R + x;
        has = 1u | (x < wo ? 2u : 0u);
        if (j + 1 < ny) has |= has << 2;
        unsigned bx = (x_edge(g, 0, x) ? 1u : 0u) | (x_edge(g, 1, x) ? 2u : 0u);
        bnd = k == 0 || k == g.nz - 1 ? 15u
              : (j == 0 || j == ny - 1 ? 3u : bx) | ((j + 1 == ny - 1 ? 3u : bx) << 2);
      };
      // r minus the products with the plane below: FP32 an item per thread (the
      // points share the lines' loads), FP64 a point per thread (a product holds
      // a warp's FP64 unit for 64 cycles, so the points go to different warps;
      // the 16^3 V-cycle took 142 us with items, 133 with points, and the 32^3
      // FP32 one 90 instead of 75)
      if constexpr (sizeof(T) == 4) {
        for (int t = tid; t < items; t += blockDim.x) {
          locate(t);
          const T* rr = r + pi;
          T s00 = rr[0], s01 = has & 2u ? rr[we] : T(0);
          T s10 = has & 4u ? rr[row] : T(0), s11 = has & 8u ? rr[row + we] : T(0);
          if (!first && k > 0) {
            const T* ln = plane_of(k - 1) + j * pitch + x;   // line j - 1
            T l[4], e[4], od[4], rt[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const bool in = u < 3 || (has & 4u);
              l[u] = in ? ln[odd - R] : T(0);
              e[u] = in ? ln[R] : T(0);
              od[u] = in ? ln[odd] : T(0);
              rt[u] = in ? ln[2 * R] : T(0);
              ln += pitch;
            }
#pragma unroll
            for (int u = 0; u < 3; ++u) {
              s00 = tail_line(P.c, u - 2, l[u], e[u], od[u], s00);
              s01 = tail_line(P.c, u - 2, e[u], od[u], rt[u], s01);
              s10 = tail_line(P.c, u - 2, l[u + 1], e[u + 1], od[u + 1], s10);
              s11 = tail_line(P.c, u - 2, e[u + 1], od[u + 1], rt[u + 1], s11);
            }
          }
          sp[4 * t] = s00;
          sp[4 * t + 1] = s01;
          sp[4 * t + 2] = s10;
          sp[4 * t + 3] = s11;
        }
      } else {
        for (int t4 = tid; t4 < 4 * items; t4 += blockDim.x) {
          const int cl = (t4 >= items) + (t4 >= 2 * items) + (t4 >= 3 * items);
          const int t = t4 - cl * items, xo = cl & 1, yo = cl >> 1;
          locate(t);
          if (!((has >> cl) & 1u)) continue;
          T acc = r[pi + yo * row + xo * we];
          if (!first && k > 0) {
            // x - 1, x, x + 1 on the lines before, of and after the point
            const T* m = plane_of(k - 1) + (j + yo) * pitch + x + (xo ? odd : R);
            const T* l = m + (xo ? R - odd : odd - 2 * R);
            T l0[3], l1[3], l2[3];
  #pragma unroll
            for (int u = 0; u < 3; ++u) {
              l0[u] = l[u * pitch];
              l1[u] = m[u * pitch];
              l2[u] = l[u * pitch + R];
            }
  #pragma unroll
            for (int u = 0; u < 3; ++u) acc = tail_line(P.c, u - 2, l0[u], l1[u], l2[u], acc);
          }
          sp[4 * t + cl] = acc;
        }
        if (tid < items) locate(tid);
      }
      __syncthreads();
      unsigned steps = op.steps;
      for (int s = 0; s < op.nsteps; ++s, steps >>= 2) {
        const int xo = steps & 1, yo = (steps >> 1) & 1, cl = steps & 3;
        const int dm = yo * pitch + xo * (odd - R), dl = xo ? R - odd : odd - 2 * R;
        for (int t = tid; t < items; t += blockDim.x) {
          if (items > (int)blockDim.x) locate(t);
          if (!((has >> cl) & 1u)) continue;
          // x-1, x, x+1 on the lines before, of and after the point
          T* m = zb + dm;
          const T* l = m + dl;
          T acc = sp[4 * t + cl];
          const T a0 = l[-pitch], a1 = m[-pitch], a2 = l[R - pitch];
          const T c0 = l[0], c2 = l[R];
          const T b0 = l[pitch], b1 = m[pitch], b2 = l[R + pitch];
          T u0[3], u1[3], u2[3];   // the plane above
          const bool above = !first && k + 1 < g.nz;
          if (above) {
#pragma unroll
            for (int u = 0; u < 3; ++u) {
              const int o = plane + (u - 1) * pitch;
              u0[u] = l[o];
              u1[u] = m[o];
              u2[u] = l[o + R];
            }
          }
          acc = tail_line(P.c, -1, a0, a1, a2, acc);
          acc = fma(-P.c.a[4], c2, fma(-P.c.a[2], c0, acc));
          acc = tail_line(P.c, 1, b0, b1, b2, acc);
          if (above) {
#pragma unroll
            for (int u = 0; u < 3; ++u) acc = tail_line(P.c, u, u0[u], u1[u], u2[u], acc);
          }
          if ((bnd >> cl) & 1u) pad_slot(*m, acc);
          T u[1] = {acc};
          if (diag) u[0] = acc / diag[pi + yo * row + xo * we];
          else div_diag<T, 1>(u);
          *m = u[0];
        }
        __syncthreads();
      }
    } else {
      // transfers with the next level: coarse point (I, J, K) <-> (2I, 2J, 2K)
      const TailLevel<T>& C = P.lev[op.level + 1];
      const int cf = first_plane(op.level + 1, rank);
      const int ce = min(first_plane(op.level + 1, rank + 1), C.g.nz);
      const int crow = C.g.we + C.g.wo;
      for (unsigned t = tid; t < (unsigned)(max(ce - cf, 0) * C.g.ny * g.we); t += blockDim.x) {
        const unsigned q = L.we.div(t), x = t - q * L.we.d;   // g.we = coarse nx * R
        const unsigned ip = C.ny.div(q), J = q - ip * C.ny.d;
        const int K = cf + (int)ip, k = 2 * K, j = 2 * (int)J;
        const unsigned I = x / (unsigned)R, rr = x - I * R;
        const unsigned cx = (I >> 1) * R + rr;   // element of its coarse line part
        if (op.kind == kTailRestrict) {
          T acc = r[((k - f) * g.ny + j) * row + x];
          const T d = L.diag ? sm[L.d + ((k - f) * g.ny + j) * row + x] : (T)kDiag;
#pragma unroll
          for (int dz = -1; dz <= 1; ++dz) {
            if (k + dz < 0 || k + dz >= g.nz) continue;
            const T* ln = plane_of(k + dz) + j * L.pitch + x;
#pragma unroll
            for (int u = 0; u < 3; ++u, ln += L.pitch) {
              if (dz == 0 && u == 1) {
                acc = fma(-P.c.a[2], ln[L.odd - R], acc);
                acc = fma(-d, ln[R], acc);
                acc = fma(-P.c.a[4], ln[L.odd], acc);
                if (j == 0 || j == g.ny - 1 || k == 0 || k == g.nz - 1 || x_edge(g, 0, x))
                  pad_slot(ln[R], acc);
              } else {
                acc = tail_line(P.c, u - 1 + dz, ln[L.odd - R], ln[R], ln[L.odd], acc);
              }
            }
          }
          sm[C.r + q * crow + cx + ((I & 1) ? C.g.we : 0)] = acc;
        } else {
          z[(k - f) * L.plane + (j + 1) * L.pitch + R + x] +=
              sm[C.z + (int)ip * C.plane + ((int)J + 1) * C.pitch + cx + ((I & 1) ? C.odd : R)];
        }
      }
    }
    if (op.cluster) tail_barrier();
    else __syncthreads();
  }

  const TailLevel<T>& L = P.lev[0];
  const int f = first_plane(0, rank), fe = min(first_plane(0, rank + 1), L.g.nz);
  for (unsigned t = tid; t < (unsigned)(max(fe - f, 0) * L.g.ny * L.g.we); t += blockDim.x) {
    const unsigned q = L.we.div(t), x = t - q * L.we.d;
    const unsigned ip = L.ny.div(q), j = q - ip * L.ny.d;
    const T* ln = sm + L.z + ip * L.plane + (j + 1) * L.pitch + x;
    P.z[line_base(L.g, 0, j, f + ip) + x] = ln[L.g.R];
    if ((int)x < L.g.wo) P.z[line_base(L.g, 1, j, f + ip) + x] = ln[L.odd];
  }
  if (rank == 0)   // padding rows (identity)
    for (int c = 0; c < kColours; ++c)
      for (unsigned p = L.g.off[c] + L.g.cnt[c] + tid; p < L.g.end[c]; p += blockDim.x)
        P.z[p] = P.given ? fma(T(-0.0), ld_dep(P.z + p), ld_dep(P.r + p)) : ld_dep(P.r + p);
}

static int tail_planes(int nz, int ctas) {   // planes per CTA of the first level
  return std::max(2, ((nz + ctas - 1) / ctas + 1) / 2 * 2);
}
// Fills P for the V-cycle from `level` down, or for `sweeps` > 0 sweeps on it;
// false if it does not fit.
template <typename T>
static bool tail_plan(const hpg_problem* h, int level, int R, int sweeps, bool from_zero,
                      int ctas, TailParams<T>& P) {
  P.nlev = sweeps ? 1 : h->nlev - level;
  P.given = sweeps && !from_zero;
  const Geom& top = h->lev[level].g;
  P.ppc = tail_planes(top.nz, ctas);
  P.ctas = (top.nz + P.ppc - 1) / P.ppc;
  P.c = make_coef<T>(h->beta);
  long long off = 0;
  for (int l = 0; l < P.nlev; ++l) {
    const Level& L = h->lev[level + l];
    TailLevel<T>& t = P.lev[l];
    t.g = make_sgeom(L.g, R);
    if (t.g.we >= (1 << 14) || t.g.ny >= (1 << 14)) return false;
    t.we = FastDiv(t.g.we);
    t.ny = FastDiv(t.g.ny);
    t.he = FastDiv(t.g.he);
    t.pitch = t.g.we + t.g.wo + 3 * R;
    t.odd = t.g.we + 2 * R;
    t.plane = (t.g.ny + 2) * t.pitch;
    t.diag = level_diag<T>(L);
    const long long planes = (P.ppc + (1 << l) - 1) >> l;
    const long long rows = planes * t.g.ny * (t.g.we + t.g.wo);
    t.z = (int)off;
    off += (planes + 1) * t.plane;   // one more: a copy of the next CTA's first plane
    t.r = (int)off;
    off += rows;
    t.d = (int)off;
    if (t.diag) off += rows;
    if (off * (long long)sizeof(T) > (long long)kTailSmem) return false;
  }
  P.sp = (int)off;
  const int most = P.ppc / 2 * P.lev[0].g.he * P.lev[0].g.we;   // items of a stage
  off += 4LL * most;
  P.threads = std::min(kTailThreads, std::max(64, ((sizeof(T) == 8 ? 4 : 1) * most + 31) / 32 * 32));
  P.elems = (int)off;
  if (off * (long long)sizeof(T) > (long long)kTailSmem || off >= (1 << 16)) return false;
  // the operations.  A cluster barrier follows an operation whose values other
  // CTAs read next; a restriction and the last stage of a level are followed by
  // operations on the CTA's own planes only.
  bool ok = true;
  P.nops = 0;
  auto push = [&](TailOp op) {
    if (P.nops < kTailOps) P.op[P.nops++] = op;
    else ok = false;
  };
  auto sweep = [&](int l, bool zero) {
    const bool odd = P.lev[l].g.dO > 0;
    const unsigned char lv = (unsigned char)l;
    // (y odd, x odd) = 11, 10, 01, 00 are the colours 0 1 2 3 (4 5 6 7)
    if (odd) push({kTailStage, lv, 1, zero, 0x1B, 4, 1});
    push({kTailStage, lv, 0, zero && !odd, 0x391B, 7, 1});
    if (odd) push({kTailStage, lv, 1, 0, 0xE4, 4, 1});
  };
  for (int i = 0; i < sweeps; ++i) sweep(0, from_zero && i == 0);
  for (int l = 0; l + 1 < P.nlev; ++l) {
    for (int i = 0; i < h->pre; ++i) sweep(l, i == 0);
    push({kTailRestrict, (unsigned char)l, 0, 0, 0, 0, 0});
  }
  if (!sweeps) sweep(P.nlev - 1, true);
  for (int l = P.nlev - 2; l >= 0; --l) {
    P.op[P.nops - 1].cluster = 0;
    push({kTailProlong, (unsigned char)l, 0, 0, 0, 0, 1});
    for (int i = 0; i < h->post; ++i) sweep(l, false);
  }
  if (ok) P.op[P.nops - 1].cluster = 1;   // no CTA leaves while others read its memory
  return ok;
}

// Largest cluster the kernel is launched with on h's device, asked once.
template <typename T>
static int tail_ctas(hpg_problem* h, int* ctas) {
  int& known = h->tail_ctas[sizeof(T) == 8 ? 0 : 1];
  if (known == 0) {
    auto kern = vcycle_tail_kernel<T>;
    HPG_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kTailSmem));
    HPG_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)kTailCtas);
    cfg.blockDim = dim3((unsigned)kTailThreads);
    cfg.dynamicSmemBytes = kTailSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)kTailCtas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    known = n > 0 ? kTailCtas : kTailPortableCtas;
  }
  *ctas = known;
  return HPG_OK;
}

template <typename T>
static int tail_t(hpg_problem* h, int level, int R, const T* r, T* z, int sweeps,
                  bool from_zero, bool c0_done, cudaStream_t s) {
  const Level& top = h->lev[level];
  TailParams<T> P;
  int most_ctas = 0;
  const int prc = tail_ctas<T>(h, &most_ctas);
  if (prc) return prc;
  const long long most = sizeof(T) == 8 ? (sweeps ? kTailSweepPoints64 : kTailPoints64)
                                        : (sweeps ? kTailSweepPoints32 : kTailPoints32);
  if ((long long)tail_planes(top.g.nz, most_ctas) * top.g.nx * top.g.ny * R > most)
    return HPG_ERR_UNSUPPORTED;
  if (!tail_plan(h, level, R, sweeps, from_zero, most_ctas, P)) return HPG_ERR_UNSUPPORTED;
  P.r = r;
  P.z = z;
  auto kern = vcycle_tail_kernel<T>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)P.ctas);
  cfg.blockDim = dim3((unsigned)P.threads);
  cfg.dynamicSmemBytes = ((size_t)P.elems * sizeof(T) + 15) / 16 * 16;
  cfg.stream = s;
  const int prec = sizeof(T) == 8 ? HPG_FP64 : HPG_FP32;
  // colour phases of the first level (what the profile counts); the lower
  // levels' operations are noted without a time of their own
  auto phases = [&](int l, int count) {
    int n = 0, m = 0;
    for (int c = 0; c < kColours; ++c) {
      n += h->lev[l].cnt[c] > 0;
      m += c < kColours - 1 && h->lev[l].cnt[c] > 0;
    }
    return count * (n + m);
  };
  const int last = h->nlev - 1;
  const int rc = launch(h, K_GS, level, prec, 2.0 * top.n * R * sizeof(T), s,
                        "vcycle_tail_kernel", [&] {
    cudaLaunchAttribute attr[2];
    int na = 0;
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = (unsigned)P.ctas;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
    if (h->pdl_enabled && h->pdl_next && !h->profiling) {
      attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[na].val.programmaticStreamSerializationAllowed = 1;
      ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, kern, P);
  }, phases(level, sweeps ? sweeps : level == last ? 1 : h->pre + h->post) - (c0_done ? 1 : 0));
  if (rc || sweeps) return rc;
  for (int l = level; l < last; ++l) {
    prof_note(h, K_RESTRICT, l, prec, 1);
    prof_note(h, K_PROLONG, l, prec, 1);
    prof_note(h, K_GS, l + 1, prec, phases(l + 1, l + 1 == last ? 1 : h->pre + h->post));
  }
  return HPG_OK;
}
int launch_vcycle_tail(hpg_problem* h, int level, int R, const float* r, float* z, bool c0_done,
                       cudaStream_t s) {
  return tail_t<float>(h, level, R, r, z, 0, true, c0_done, s);
}
int launch_vcycle_tail(hpg_problem* h, int level, int R, const double* r, double* z, bool c0_done,
                       cudaStream_t s) {
  return tail_t<double>(h, level, R, r, z, 0, true, c0_done, s);
}

int launch_small_sweeps(hpg_problem* h, int level, const float* r, float* z, int sweeps,
                        bool from_zero, cudaStream_t s) {
  return tail_t<float>(h, level, 1, r, z, sweeps, from_zero, false, s);
}
int launch_small_sweeps(hpg_problem* h, int level, const double* r, double* z, int sweeps,
                        bool from_zero, cudaStream_t s) {
  return tail_t<double>(h, level, 1, r, z, sweeps, from_zero, false, s);
}

}  // namespace hpg
