// Frozen electric potential (Eq. 4-5 with the Dirichlet surface value of
// Sec. 2) by Jacobi-preconditioned conjugate gradients, accurate to FP64.
//
// For a pore cell P the discrete equation is
//   sum_f T_f (psi_nb - psi_P) - kdx2 psi_P = 0,
// T_f = 1 towards a pore neighbour or the inlet feed (psi = 0), 2 towards a
// solid face (psi = psi_s at half a cell), 0 at the outlet and lateral walls;
// kdx2 = (dx / lambda_D)^2 screens the field (Debye-Hueckel linearisation of
// Eq. 4-5; 0 gives Laplace).  With the coupling of Eq. 3-5 on, the right-hand
// side also carries the charge term dx^2 rho_e / (eps_r eps_0) of every pore
// cell (Eq. 5 from the current concentrations).  The linear modes run as FP32
// corrections of an FP64 residual (k_psi_refine); the nonlinear mode, and what
// the corrections cannot solve, as an FP64 iteration whose scalars stay on the
// device, its convergence flag polled every few iterations.
#include <cmath>

#include "cdi_internal.cuh"

using namespace cdi;

namespace {

struct Geo {
  int nx, ny, nz, dim, walls;
  long long N;
};

// Face f of pore cell (x,y,z): 0 pore neighbour (index in *nb), 1 solid,
// 2 inlet feed, 3 no flux (outlet or lateral wall).
__device__ __forceinline__ int face_kind(const Geo &g, const NFlag *fl, long long P, int x,
                                         int y, int z, int f, long long *nb) {
  const int a = f >> 1;
  const int s = (f & 1) ? -1 : 1;
  if (a == 0) {
    if (x + s < 0) return 2;
    if (x + s >= g.nx) return 3;
    if ((fl[P] >> (kFaceBit + f)) & 1) return 1;
    *nb = P + s;
    return 0;
  }
  int Y = y, Z = z;
  if (a == 1) {
    Y = y + s;
    if (Y < 0 || Y >= g.ny) {
      if (g.walls) return 3;
      Y = (Y + g.ny) % g.ny;
    }
  } else {
    Z = z + s;
    if (Z < 0 || Z >= g.nz) {
      if (g.walls) return 3;
      Z = (Z + g.nz) % g.nz;
    }
  }
  if ((fl[P] >> (kFaceBit + f)) & 1) return 1;
  *nb = ((long long)Z * g.ny + Y) * g.nx + x;
  return 0;
}

__device__ __forceinline__ void coords(const Geo &g, long long P, int &x, int &y, int &z) {
  const long long row = P / g.nx;
  x = (int)(P - row * g.nx);
  z = (int)(row / g.ny);
  y = (int)(row - (long long)z * g.ny);
}

// diag, right-hand side, x = 0, r = b, z = r / diag, p = z; rz and b.b.
__global__ void __launch_bounds__(kRedThreads)
    k_cg_setup(Geo g, const NFlag *__restrict__ fl, double kdx2, double psi_s,
               const double *__restrict__ src, double tol,
               double *__restrict__ x, double *__restrict__ r, double *__restrict__ p,
               double *__restrict__ diag, double *__restrict__ part, unsigned int *counter,
               double *scal) {
  __shared__ double sm[2 * 32];
  double v[2] = {0.0, 0.0};
  for (long long P = blockIdx.x * (long long)blockDim.x + threadIdx.x; P < g.N;
       P += (long long)gridDim.x * blockDim.x) {
    x[P] = 0.0;
    if (fl[P] & 1) {
      r[P] = 0.0;
      p[P] = 0.0;
      diag[P] = 1.0;
      continue;
    }
    int cx, cy, cz;
    coords(g, P, cx, cy, cz);
    double dg = kdx2, b = src ? src[P] : 0.0;
    for (int f = 0; f < 2 * g.dim; f++) {
      long long nb;
      const int k = face_kind(g, fl, P, cx, cy, cz, f, &nb);
      if (k == 0 || k == 2) dg += 1.0;
      if (k == 1) {
        dg += 2.0;
        b += 2.0 * psi_s;
      }
    }
    diag[P] = dg;
    r[P] = b;
    p[P] = b / dg;
    v[0] += b * (b / dg);
    v[1] += b * b;
  }
  block_reduce<2>(v, sm, OpSum(), 0.0);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = v[0];
    part[gridDim.x + blockIdx.x] = v[1];
  }
  if (last_block(counter, gridDim.x)) {
    combine_partials<2>(part, gridDim.x, v, sm, OpSum(), 0.0);
    if (threadIdx.x == 0) {
      scal[S_CG_RZ] = v[0];
      scal[S_CG_BB] = v[1];
      scal[S_CG_RR] = v[1];
      scal[S_CG_REL] = v[1] > 0.0 ? 1.0 : 0.0;
      scal[S_CG_DONE] = v[1] > 0.0 ? 0.0 : 1.0;
      scal[S_CG_TOL] = tol;
      scal[S_CG_IT] = 0.0;
      *counter = 0;
    }
  }
}

// One Newton step of the nonlinear Poisson-Boltzmann equation (Eq. 4 with
// the Boltzmann charge of Eq. 9 for a 1:1 salt; Eq. 10 in 1D), per pore cell
//   F_P(psi) = (A0 psi)_P - b_P + kdx2 V_T sinh(psi_P / V_T) = 0,
// A0 and b the face rules above.  Newton solves
//   (A0 + kdx2 cosh(psi / V_T)) psi' = b + kdx2 (psi cosh(psi / V_T) - V_T sinh(psi / V_T))
// by the CG below, warm-started at psi' = psi, so its first residual is -F.
// This kernel forms F (F.F and b.b into S_PB_FF / S_PB_BB: the Newton test),
// the CG's diagonal and its start (r = -F, p = r / diag, rz, and the
// right-hand side's b.b for the CG's relative residual).  psi is only read.
__global__ void __launch_bounds__(kRedThreads)
    k_pb_setup(Geo g, const NFlag *__restrict__ fl, double kdx2, double psi_s, double vt,
               double tol, const double *__restrict__ psi, double *__restrict__ r,
               double *__restrict__ p, double *__restrict__ diag, double *__restrict__ part,
               unsigned int *counter, double *scal) {
  __shared__ double sm[4 * 32];
  double v[4] = {0.0, 0.0, 0.0, 0.0};  // rz, rhs.rhs, F.F, b.b
  for (long long P = blockIdx.x * (long long)blockDim.x + threadIdx.x; P < g.N;
       P += (long long)gridDim.x * blockDim.x) {
    if (fl[P] & 1) {
      r[P] = 0.0;
      p[P] = 0.0;
      diag[P] = 1.0;
      continue;
    }
    int cx, cy, cz;
    coords(g, P, cx, cy, cz);
    double t = 0.0, b = 0.0, off = 0.0;
    for (int f = 0; f < 2 * g.dim; f++) {
      long long nb;
      const int k = face_kind(g, fl, P, cx, cy, cz, f, &nb);
      if (k == 0) {
        t += 1.0;
        off += psi[nb];
      } else if (k == 2) {
        t += 1.0;
      } else if (k == 1) {
        t += 2.0;
        b += 2.0 * psi_s;
      }
    }
    const double x = psi[P], ph = x / vt;
    const double sh = sinh(ph), ch = cosh(ph);
    const double F = t * x - off - b + kdx2 * vt * sh;
    const double dg = t + kdx2 * ch;
    const double rhs = b + kdx2 * (x * ch - vt * sh);
    diag[P] = dg;
    r[P] = -F;
    p[P] = -F / dg;
    v[0] += F * (F / dg);
    v[1] += rhs * rhs;
    v[2] += F * F;
    v[3] += b * b;
  }
  block_reduce<4>(v, sm, OpSum(), 0.0);
  if (threadIdx.x == 0)
    for (int k = 0; k < 4; k++) part[k * gridDim.x + blockIdx.x] = v[k];
  if (last_block(counter, gridDim.x)) {
    combine_partials<4>(part, gridDim.x, v, sm, OpSum(), 0.0);
    if (threadIdx.x == 0) {
      scal[S_CG_RZ] = v[0];
      scal[S_CG_BB] = v[1];
      scal[S_CG_RR] = v[2];
      scal[S_CG_REL] = v[1] > 0.0 ? sqrt(v[2] / v[1]) : 0.0;
      scal[S_CG_DONE] = (v[1] > 0.0 && v[2] > 0.0) ? 0.0 : 1.0;
      scal[S_CG_TOL] = tol;
      scal[S_CG_IT] = 0.0;
      scal[S_PB_FF] = v[2];
      scal[S_PB_BB] = v[3];
      *counter = 0;
    }
  }
}

// q = A p and p.q; alpha = rz / p.q.
__global__ void __launch_bounds__(kRedThreads)
    k_cg_spmv(Geo g, const NFlag *__restrict__ fl, const double *__restrict__ p,
              const double *__restrict__ diag, double *__restrict__ q,
              double *__restrict__ part, unsigned int *counter, double *scal) {
  if (scal[S_CG_DONE] != 0.0) return;
  __shared__ double sm[32];
  double v[1] = {0.0};
  for (long long P = blockIdx.x * (long long)blockDim.x + threadIdx.x; P < g.N;
       P += (long long)gridDim.x * blockDim.x) {
    if (fl[P] & 1) {
      q[P] = 0.0;
      continue;
    }
    int cx, cy, cz;
    coords(g, P, cx, cy, cz);
    double off = 0.0;
    for (int f = 0; f < 2 * g.dim; f++) {
      long long nb;
      if (face_kind(g, fl, P, cx, cy, cz, f, &nb) == 0) off += p[nb];
    }
    const double qv = diag[P] * p[P] - off;
    q[P] = qv;
    v[0] += p[P] * qv;
  }
  block_reduce<1>(v, sm, OpSum(), 0.0);
  if (threadIdx.x == 0) part[blockIdx.x] = v[0];
  if (last_block(counter, gridDim.x)) {
    combine_partials<1>(part, gridDim.x, v, sm, OpSum(), 0.0);
    if (threadIdx.x == 0) {
      scal[S_CG_PQ] = v[0];
      scal[S_CG_ALPHA] = v[0] != 0.0 ? scal[S_CG_RZ] / v[0] : 0.0;
      *counter = 0;
    }
  }
}

// x += alpha p, r -= alpha q, z = r / diag (into q); beta = rz' / rz.
__global__ void __launch_bounds__(kRedThreads)
    k_cg_update(long long N, const NFlag *__restrict__ fl, double *__restrict__ x,
                double *__restrict__ r, const double *__restrict__ p, double *__restrict__ q,
                const double *__restrict__ diag, double *__restrict__ part,
                unsigned int *counter, double *scal) {
  if (scal[S_CG_DONE] != 0.0) return;
  __shared__ double sm[2 * 32];
  const double alpha = scal[S_CG_ALPHA];
  double v[2] = {0.0, 0.0};
  for (long long P = blockIdx.x * (long long)blockDim.x + threadIdx.x; P < N;
       P += (long long)gridDim.x * blockDim.x) {
    if (fl[P] & 1) continue;
    x[P] += alpha * p[P];
    const double rv = r[P] - alpha * q[P];
    r[P] = rv;
    const double zv = rv / diag[P];
    q[P] = zv;
    v[0] += rv * zv;
    v[1] += rv * rv;
  }
  block_reduce<2>(v, sm, OpSum(), 0.0);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = v[0];
    part[gridDim.x + blockIdx.x] = v[1];
  }
  if (last_block(counter, gridDim.x)) {
    combine_partials<2>(part, gridDim.x, v, sm, OpSum(), 0.0);
    if (threadIdx.x == 0) {
      const double rz_old = scal[S_CG_RZ];
      scal[S_CG_BETA] = rz_old != 0.0 ? v[0] / rz_old : 0.0;
      scal[S_CG_RZ] = v[0];
      scal[S_CG_RR] = v[1];
      const double rel = sqrt(v[1] / scal[S_CG_BB]);
      scal[S_CG_REL] = rel;
      scal[S_CG_IT] += 1.0;
      if (rel < scal[S_CG_TOL] || v[0] == 0.0) scal[S_CG_DONE] = 1.0;
      *counter = 0;
    }
  }
}

// p = z + beta p.
__global__ void k_cg_dir(long long N, double *__restrict__ p, const double *__restrict__ zq,
                         const double *__restrict__ scal) {
  if (scal[S_CG_DONE] != 0.0) return;
  const double beta = scal[S_CG_BETA];
  for (long long P = blockIdx.x * (long long)blockDim.x + threadIdx.x; P < N;
       P += (long long)gridDim.x * blockDim.x)
    p[P] = zq[P] + beta * p[P];
}

// ---------------------------------------------------------------------------
// The linear potential by iterative refinement: the residual b - A x and the
// sums x += d in FP64, the corrections A d = r by the same Jacobi-PCG in FP32
// to a relative 1e-4, repeated until the FP64 residual itself (not a
// recurrence of it) is below tol.  One cooperative launch, vectors by pore
// rank.
//
// Why: at 2 FP64 operations a clock and SM an FP64 iteration is bound by its
// arithmetic (14 operations a cell and a division), and as three launches over
// the whole lattice with 64-bit coordinate divisions it took far longer; an
// FP32 iteration moves 64 bytes a cell, out of L2 up to 128^3.  The direction
// update is folded into the product (a neighbour's new p from its z and old
// p), which leaves two grid barriers an iteration.  128^3 Laplace: 33.7 ->
// 6.0 ms (18 us an iteration, 9 us at 64^3), its error against 64 bits 8.6e-13
// -> 3e-13.  Of that, pair sums and FP32 scalars 8.5 -> 5.8 ms, (z, p) records,
// 16-bit links and two cells a thread at a time 9.0 -> 8.3 ms.
// ---------------------------------------------------------------------------
struct PsiArgs {
  const NFlag *fl;    // per rank face flags
  const int *lat;     // lateral neighbour ranks (read where latd does not hold them)
  const short *latd;  // 16-bit lateral differences per rank
  const int *latb;    // their bases per tile of 31 ranks
  const int *cells;
  const double *src;  // lattice order, or null
  int n, walls, max_iter;
  double kdx2, psi_s, tol;
  double *x;          // rank order
  float *f;           // 7 n: (z, p) in two buffers, r, d, q
  uint16_t *meta;     // n: see psi_meta
  double *psi;        // lattice order, zero at solid cells
  double *part, *scal;
  unsigned *counter;
};

// Open (pore) faces of a pore cell in bits 8.., the integer part of its
// diagonal (1 a pore or inlet face, 2 a solid one) below.
template <int DIM> __device__ __forceinline__ unsigned psi_meta(unsigned f, int walls, int &solids) {
  unsigned t = 0, open = 0;
  solids = 0;
#pragma unroll
  for (int fc = 0; fc < 2 * DIM; fc++) {
    const bool solid = (f >> (kFaceBit + fc)) & 1u, edge = (f >> (kEdgeBit + fc)) & 1u;
    const bool no_flux = edge && (fc == 0 || (fc > 1 && walls));
    if (fc == 1 && edge) {  // inlet feed
      t += 1;
    } else if (solid && !no_flux) {
      t += 2;
      solids++;
    } else if (!no_flux) {
      t += 1;
      open |= 1u << fc;
    }
  }
  return t | open << 8;
}

// Ranks across the faces of rank r (r itself across a closed one, so that the
// loads need no branch).
template <int DIM>
__device__ __forceinline__ void psi_ranks(const PsiArgs &a, unsigned m, int r, int (&q)[2 * DIM]) {
  constexpr int NL = 2 * DIM - 2;
  const int t = r / 31;
  int base[NL], diff[NL];
  if constexpr (DIM == 3) {
    const int4 b = reinterpret_cast<const int4 *>(a.latb)[t];
    const short4 v = reinterpret_cast<const short4 *>(a.latd)[r];
    base[0] = b.x; base[1] = b.y; base[2] = b.z; base[3] = b.w;
    diff[0] = v.x; diff[1] = v.y; diff[2] = v.z; diff[3] = v.w;
  } else {
    const int2 b = reinterpret_cast<const int2 *>(a.latb)[t];
    const short2 v = reinterpret_cast<const short2 *>(a.latd)[r];
    base[0] = b.x; base[1] = b.y;
    diff[0] = v.x; diff[1] = v.y;
  }
  bool wide = false;
#pragma unroll
  for (int f = 0; f < 2 * DIM; f++) {
    const int to = f < 2 ? r + (f == 0 ? 1 : -1) : r + base[f < 2 ? 0 : f - 2] + diff[f < 2 ? 0 : f - 2];
    q[f] = (m >> (8 + f)) & 1u ? to : r;
    if (f >= 2) wide |= diff[f < 2 ? 0 : f - 2] == kLatWide;
  }
  if (wide)
#pragma unroll
    for (int f = 2; f < 2 * DIM; f++)
      q[f] = (m >> (8 + f)) & 1u ? a.lat[(size_t)(f - 2) * a.n + r] : r;
}

// s + c += v (the rounding errors of s gathered in c).
__device__ __forceinline__ void sum_acc(float v, float &s, float &c) {
  const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
  c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b)));
  s = t;
}

template <int DIM> __global__ void __launch_bounds__(kGridThreads) k_psi_refine(PsiArgs a) {
  extern __shared__ double sm[];  // 3 rows of a value a warp (GridBarrier)
  __shared__ float2 tot[kGridSums];
  __shared__ double tot64[2];
  __shared__ float dia[16], idia[16];
  const int first = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  const size_t n = (size_t)a.n;
  // records (z, p), so that a neighbour is one load
  float2 *w0 = (float2 *)a.f, *w1 = w0 + n;
  float *rr = a.f + 4 * n, *d = rr + n, *q = d + n;
  GridBarrier bar{a.counter, a.part, sm, (int)(blockDim.x >> 5), 0u, 0};
  // the norms, once a cycle, stay FP64: they decide when to stop, and squares
  // of a small potential's residuals leave FP32's range
  auto add64 = [&](int k, double v) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) sm[k * bar.row + (threadIdx.x >> 5)] = v;
  };
  if (threadIdx.x < 16) {
    const double v = a.kdx2 + threadIdx.x;
    dia[threadIdx.x] = (float)v;
    idia[threadIdx.x] = v > 0.0 ? (float)(1.0 / v) : 0.f;
  }
  double v = 0.0;
  for (int r = first; r < a.n; r += stride) {
    int solids;
    a.meta[r] = (uint16_t)psi_meta<DIM>(a.fl[r], a.walls, solids);
    const double b = 2.0 * solids * a.psi_s + (a.src ? a.src[a.cells[r]] : 0.0);
    a.x[r] = 0.0;
    v += b * b;
  }
  add64(0, v);
  if (!grid_totals(bar, tot64, 1)) return grid_give_up(a.scal + S_CG_ALPHA);
  const double bb = tot64[0];
  double rel = bb > 0.0 ? 1.0 : 0.0, scale = bb > 0.0 ? sqrt(a.n / bb) : 1.0;
  int it = 0;
  bool done = bb == 0.0;

  for (int cycle = 0; !done; cycle++) {
    // r = b - A x, its FP32 image scaled to a mean square of about 1
    v = 0.0;
    float zs = 0.f, zc = 0.f;
    for (int r = first; r < a.n; r += stride) {
      const unsigned m = a.meta[r];
      int solids;
      psi_meta<DIM>(a.fl[r], a.walls, solids);
      double res = 2.0 * solids * a.psi_s + (a.src ? a.src[a.cells[r]] : 0.0);
      if (cycle > 0) {
        int k[2 * DIM];
        psi_ranks<DIM>(a, m, r, k);
#pragma unroll
        for (int f = 0; f < 2 * DIM; f++)
          if ((m >> (8 + f)) & 1u) res += a.x[k[f]];
        res -= (a.kdx2 + (m & 255u)) * a.x[r];
      }
      v += res * res;
      const float rv = (float)(res * scale), zv = rv * idia[m & 255u];
      rr[r] = rv;
      w0[r] = make_float2(zv, 0.f);
      d[r] = 0.f;
      sum_acc(rv * zv, zs, zc);
    }
    add64(0, v);
    add64(1, (double)zs + (double)zc);
    if (!grid_totals(bar, tot64, 2)) return grid_give_up(a.scal + S_CG_ALPHA);
    const double rr64 = tot64[0], old = rel;
    float rz = (float)tot64[1];
    rel = sqrt(rr64 / bb);
    if (rel < a.tol || rr64 == 0.0) {
      done = true;
      break;
    }
    if (it >= a.max_iter || (cycle > 0 && !(rel < 0.5 * old))) break;

    const double eta = fmin(fmax(0.3 * a.tol / rel, 1e-4), 0.1);
    const float target = (float)(eta * eta * (rr64 * scale * scale));
    // (the iteration's scalars in FP32 too: an FP64 division is microseconds)
    float rr32 = 0.f, beta = 0.f;
    while (it < a.max_iter) {
      // q = A p for p = z + beta p; p . q.  Two cells of a thread at a time:
      // the pass is bound by the latency of its two levels of loads.
      float s = 0.f, c = 0.f;
      for (int r = first; r < a.n; r += 2 * stride) {
        const int rs[2] = {r, min(r + stride, a.n - 1)};
        const int two = r + stride < a.n ? 2 : 1;
        unsigned m[2];
        int k[2][2 * DIM];
        float2 own[2], nb[2][2 * DIM];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          m[u] = a.meta[rs[u]];
          own[u] = w0[rs[u]];
          psi_ranks<DIM>(a, m[u], rs[u], k[u]);
        }
#pragma unroll
        for (int u = 0; u < 2; u++)
#pragma unroll
          for (int f = 0; f < 2 * DIM; f++) nb[u][f] = w0[k[u][f]];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const float pv = fmaf(beta, own[u].y, own[u].x);
          float off = 0.f;
#pragma unroll
          for (int f = 0; f < 2 * DIM; f++)
            if ((m[u] >> (8 + f)) & 1u) off += fmaf(beta, nb[u][f].y, nb[u][f].x);
          const float qv = fmaf(dia[m[u] & 255u], pv, -off);
          if (u < two) {
            q[rs[u]] = qv;
            sum_acc(pv * qv, s, c);
          }
        }
      }
      grid_add(bar, 0, s, c);
      if (!grid_totals(bar, tot, 1)) return grid_give_up(a.scal + S_CG_ALPHA);
      const float pq = tot[0].x + tot[0].y, alpha = pq != 0.f ? rz / pq : 0.f;
      // p = z + beta p, d += alpha p, r -= alpha q, z = r / diag; r . z and r . r
      float zs = 0.f, zc = 0.f, rs = 0.f, rc = 0.f;
      for (int r = first; r < a.n; r += 2 * stride) {
        const int at[2] = {r, min(r + stride, a.n - 1)};
        const int two = r + stride < a.n ? 2 : 1;
        float2 own[2];
        float qv[2], rv[2], dv[2], iv[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          own[u] = w0[at[u]];
          qv[u] = q[at[u]];
          rv[u] = rr[at[u]];
          dv[u] = d[at[u]];
          iv[u] = idia[a.meta[at[u]] & 255u];
        }
#pragma unroll
        for (int u = 0; u < 2; u++) {
          if (u >= two) continue;
          const float pv = fmaf(beta, own[u].y, own[u].x);
          const float res = fmaf(-alpha, qv[u], rv[u]), zv = res * iv[u];
          d[at[u]] = fmaf(alpha, pv, dv[u]);
          rr[at[u]] = res;
          w1[at[u]] = make_float2(zv, pv);
          sum_acc(res * zv, zs, zc);
          sum_acc(res * res, rs, rc);
        }
      }
      grid_add(bar, 0, zs, zc);
      grid_add(bar, 1, rs, rc);
      if (!grid_totals(bar, tot, 2)) return grid_give_up(a.scal + S_CG_ALPHA);
      const float next = tot[0].x + tot[0].y;
      beta = rz != 0.f ? next / rz : 0.f;
      rz = next;
      rr32 = tot[1].x + tot[1].y;
      float2 *t = w0;
      w0 = w1;
      w1 = t;
      it++;
      if (!(rr32 > target)) break;  // (a NaN also ends it: the cycle's test sees that)
    }
    // x += d
    const double unscale = 1.0 / scale;
    for (int r = first; r < a.n; r += stride) a.x[r] += (double)d[r] * unscale;
    if (!grid_totals(bar, tot, 0)) return grid_give_up(a.scal + S_CG_ALPHA);
    if (rr32 > 0.f && rr32 < 1e30f) scale *= sqrt((double)a.n / rr32);
  }
  for (int r = first; r < a.n; r += stride) a.psi[a.cells[r]] = a.x[r];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.scal[S_CG_REL] = rel;
    a.scal[S_CG_DONE] = done ? 1.0 : 0.0;
    a.scal[S_CG_IT] = it;
  }
}

// The charge term of Eq. 4 at every pore cell from Eq. 5:
// src = coef * sum_k z_k C_k, coef = F dx^2 / (eps_r eps_0) (lattice order;
// solid cells keep the 0 the caller cleared).
template <typename T>
__global__ void k_charge(int n, int ns, const int *__restrict__ cells, CViews<T> C, int4 z,
                         double coef, double *__restrict__ src) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    const int zz[4] = {z.x, z.y, z.z, z.w};
    double q = 0.0;
    for (int k = 0; k < ns; k++)
      q += zz[k] * C.v[k].at(r);
    src[cells[r]] = coef * q;
  }
}

// phi = psi / V_T of every pore rank, in the transport kernel's format.
template <typename T>
__global__ void k_phi(int n, const int *__restrict__ cells, const double *__restrict__ psi,
                      typename PhiStore<T>::type *__restrict__ phi, double inv_vt) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x)
    phi[r] = PhiStore<T>::make(psi[cells[r]] * inv_vt);
}

}  // namespace

// CG iterations (the scalars set up by k_cg_setup or k_pb_setup) until the
// device flags convergence or max_iter iterations ran; the host polls the
// flag after 8, 16, 32, ... iterations (at most 256 between polls).
static cdi_status cg_iterate(cdi_domain *d, const Geo &g, double *r, double *p, double *q,
                             const double *dg, int max_iter, bool *done) {
  int launched = 0;
  int chunk = 8;
  *done = false;
  while (launched < max_iter) {
    const int n = std::min(chunk, max_iter - launched);
    for (int k = 0; k < n; k++) {
      k_cg_spmv<<<kRedBlocks, kRedThreads, 0, d->stream>>>(g, d->d_nflags, p, dg, q, d->d_part,
                                                            d->d_counter + C_CG1, d->d_scal);
      k_cg_update<<<kRedBlocks, kRedThreads, 0, d->stream>>>(
          d->N, d->d_nflags, d->d_psi, r, p, q, dg, d->d_part, d->d_counter + C_CG2, d->d_scal);
      k_cg_dir<<<kRedBlocks, kRedThreads, 0, d->stream>>>(d->N, p, q, d->d_scal);
    }
    d->timing.kernel_launches += 3 * n;
    launched += n;
    CDI_TRY(d, cudaGetLastError(), "cg iteration");
    CDI_TRY(d, cudaMemcpyAsync(d->h_scal + S_CG_REL, d->d_scal + S_CG_REL, 4 * sizeof(double),
                               cudaMemcpyDeviceToHost, d->stream),
            "cg poll");
    CDI_TRY(d, cudaStreamSynchronize(d->stream), "cg poll");
    if (d->h_scal[S_CG_DONE] != 0.0) {
      *done = true;
      break;
    }
    chunk = std::min(chunk * 2, 256);
  }
  return CDI_OK;
}

static cdi_status finish_potential(cdi_domain *d, cudaEvent_t ev, bool done, int *iters,
                                   double *relres);

// Screened systems stay with the FP64 iteration and keep their bits, in every
// storage type.  They need fewer iterations (the condition number is below (12 +
// kdx2) / kdx2), and they are the fields that transport runs on: the face data
// of FP32 storage rounds them, and a rounding that a change in their 13th digit
// turns moves a concentration of a resolved double layer by 2e-7.  It costs
// time: 96^3, 75 iterations and 5.5 ms at kdx2 = 0.44, where refinement takes
// 1.9 ms; 158 and 11.4 ms, 3.7 ms at 0.06; 5 and 0.6 ms, 0.4 ms at the default
// screening.
constexpr double kRefineBelow = 0.05;

// The refinement above; *done says whether it reached tol.  Where it does not
// (max_iter ran out first, tol below what an FP64 residual can show, or a
// system too ill-conditioned for FP32 corrections) the caller starts over
// with the FP64 iteration, whose own residual is a recurrence.  That one gets
// all of max_iter again, since corrections may take more iterations than it
// does; the figures returned are its own, the timing counts both.
static cdi_status psi_refine(cdi_domain *d, double psi_s, double kdx2, const double *src,
                             double tol, int max_iter, bool *done) {
  *done = false;
  if (!(kdx2 < kRefineBelow)) return CDI_OK;
  const void *kern = d->dim == 2 ? (const void *)k_psi_refine<2> : (const void *)k_psi_refine<3>;
  const int n = (int)d->n_pore;
  int threads = 0;
  size_t smem = 0;
  const int blocks = n > 0 ? grid_shape(kern, n, 32, 3, &threads, &smem) : 0;
  if (blocks == 0) return CDI_OK;
  PsiArgs a;
  a.fl = d->d_cfl;
  a.lat = d->d_latnb;
  a.latd = d->d_latd;
  a.latb = d->d_latb;
  a.cells = d->d_cell_list;
  a.src = src;
  a.n = n;
  a.walls = d->walls;
  a.max_iter = max_iter;
  a.kdx2 = kdx2;
  a.psi_s = psi_s;
  a.tol = tol;
  a.x = (double *)d->d_phi;  // 8 bytes a rank; phi is formed again after the solve
  a.f = (float *)d->d_cg;    // 30 of its 32 bytes a cell
  a.meta = (uint16_t *)(a.f + 7 * (size_t)n);
  a.psi = d->d_psi;
  a.part = d->d_part;
  a.scal = d->d_scal;
  a.counter = d->d_counter + C_CG1;
  CDI_TRY(d, cudaMemsetAsync(d->d_psi, 0, (size_t)d->N * 8, d->stream), "potential reset");
  CDI_TRY(d, cudaMemsetAsync(a.counter, 0, sizeof(unsigned), d->stream), "potential barrier");
  CDI_TRY(d, cudaMemsetAsync(d->d_scal + S_CG_ALPHA, 0, sizeof(double), d->stream),
          "potential barrier");
  void *args[] = {&a};
  CDI_TRY(d, cudaLaunchCooperativeKernel(kern, dim3(blocks), dim3(threads), args, smem, d->stream),
          "potential solve");
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaMemcpyAsync(d->h_scal + S_CG_ALPHA, d->d_scal + S_CG_ALPHA, 8 * sizeof(double),
                             cudaMemcpyDeviceToHost, d->stream),
          "potential result");
  // the barrier's arrivals leave the slot that other kernels expect at 0
  CDI_TRY(d, cudaMemsetAsync(a.counter, 0, sizeof(unsigned), d->stream), "potential barrier");
  CDI_TRY(d, cudaStreamSynchronize(d->stream), "potential");
  if (d->h_scal[S_CG_ALPHA] != 0.0)
    return cdi_fail(d, CDI_ERR_CUDA, "potential solve: a grid barrier ran into its limit");
  *done = d->h_scal[S_CG_DONE] != 0.0;
  if (!*done) d->timing.psi_iters += (int64_t)d->h_scal[S_CG_IT];
  return CDI_OK;
}

cdi_status cdi_psi_solve(cdi_domain *d, double psi_s, double kdx2, const double *src,
                         double tol, int max_iter, int *iters, double *relres) {
  Geo g{d->nx, d->ny, d->nz, d->dim, d->walls, d->N};
  double *r = d->d_cg, *p = d->d_cg + d->N, *q = d->d_cg + 2 * d->N, *dg = d->d_cg + 3 * d->N;
  cudaEvent_t ev;
  cdi_timing_begin(d, &ev);
  bool done = false;
  cdi_status cs = psi_refine(d, psi_s, kdx2, src, tol, max_iter, &done);
  if (cs != CDI_OK) {
    cdi_timing_end(d, ev, PH_PSI, 0);
    return cs;
  }
  if (done) return finish_potential(d, ev, done, iters, relres);
  k_cg_setup<<<kRedBlocks, kRedThreads, 0, d->stream>>>(g, d->d_nflags, kdx2, psi_s, src, tol,
                                                         d->d_psi, r, p, dg, d->d_part,
                                                         d->d_counter + C_CG1, d->d_scal);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "cg setup");
  cs = cg_iterate(d, g, r, p, q, dg, max_iter, &done);
  if (cs != CDI_OK) return cs;
  return finish_potential(d, ev, done, iters, relres);
}

// phi = psi / V_T for the transport step, the solve's figures to the host.
static cdi_status finish_potential(cdi_domain *d, cudaEvent_t ev, bool done, int *iters,
                                   double *relres) {
  // phi keeps FP64 accuracy in both precisions (a double, or an FP32 hi/lo
  // pair): the Boltzmann factor exp(z phi) of a face turns an absolute error
  // of phi into a relative error of C.
  const double inv_vt = 1.0 / d->VT;
  if (d->prec == CDI_FP64)
    k_phi<double><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        (int)d->n_pore, d->d_cell_list, d->d_psi, (double *)d->d_phi, inv_vt);
  else
    k_phi<float><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        (int)d->n_pore, d->d_cell_list, d->d_psi, (float2 *)d->d_phi, inv_vt);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "phi");
  CDI_TRY(d, cudaMemcpyAsync(d->h_scal + S_CG_REL, d->d_scal + S_CG_REL, 4 * sizeof(double),
                             cudaMemcpyDeviceToHost, d->stream),
          "cg result");
  cdi_timing_end(d, ev, PH_PSI, 0);
  CDI_TRY(d, cudaStreamSynchronize(d->stream), "potential");
  const int it = (int)d->h_scal[S_CG_IT];
  d->timing.psi_iters += it;
  if (iters) *iters = it;
  if (relres) *relres = d->h_scal[S_CG_REL];
  return (done || d->h_scal[S_CG_DONE] != 0.0) ? CDI_OK : CDI_ERR_NOT_CONVERGED;
}

// Nonlinear Poisson-Boltzmann potential: Newton from psi = 0 (its first step
// is the screened Debye-Hueckel field), each step a CG solve warm-started at
// the current psi (k_pb_setup), until |F| <= tol |b| (b the surface terms).
// The problem is the minimum of a strictly convex energy and, psi keeping the
// sign of psi_s, Newton's iterates approach it monotonically after the first
// step.  Each CG runs to 0.1 tol of its right-hand side, at most max_iter
// iterations.  iters: the CG iterations of all steps; relres: |F| / |b|.
cdi_status cdi_psi_pb(cdi_domain *d, double psi_s, double kdx2, double tol, int max_iter,
                      int *iters, double *relres) {
  constexpr int kMaxNewton = 200;
  Geo g{d->nx, d->ny, d->nz, d->dim, d->walls, d->N};
  double *r = d->d_cg, *p = d->d_cg + d->N, *q = d->d_cg + 2 * d->N, *dg = d->d_cg + 3 * d->N;
  cudaEvent_t ev;
  cdi_timing_begin(d, &ev);
  CDI_TRY(d, cudaMemsetAsync(d->d_psi, 0, (size_t)d->N * 8, d->stream), "pb start");
  bool converged = false;
  double rel = 0.0;
  int cg_total = 0;
  for (int step = 0;; step++) {
    k_pb_setup<<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        g, d->d_nflags, kdx2, psi_s, d->VT, 0.1 * tol, d->d_psi, r, p, dg, d->d_part,
        d->d_counter + C_CG1, d->d_scal);
    d->timing.kernel_launches++;
    CDI_TRY(d, cudaGetLastError(), "pb setup");
    CDI_TRY(d, cudaMemcpyAsync(d->h_scal + S_PB_FF, d->d_scal + S_PB_FF, 2 * sizeof(double),
                               cudaMemcpyDeviceToHost, d->stream),
            "pb residual");
    CDI_TRY(d, cudaStreamSynchronize(d->stream), "pb residual");
    const double ff = d->h_scal[S_PB_FF], bb = d->h_scal[S_PB_BB];
    rel = bb > 0.0 ? std::sqrt(ff / bb) : 0.0;
    if (rel < tol) {
      converged = true;
      break;
    }
    if (step == kMaxNewton) break;
    bool done = false;
    cdi_status cs = cg_iterate(d, g, r, p, q, dg, max_iter, &done);
    if (cs != CDI_OK) return cs;
    cg_total += (int)d->h_scal[S_CG_IT];
  }
  cdi_status s = finish_potential(d, ev, true, nullptr, nullptr);
  if (s != CDI_OK) return s;
  d->timing.psi_iters += cg_total;
  if (iters) *iters = cg_total;
  if (relres) *relres = rel;
  return converged ? CDI_OK : CDI_ERR_NOT_CONVERGED;
}

// Coupled re-solve (Eq. 3-5): the charge term of the current concentrations,
// then Eq. 4 with the Laplace operator and the domain's surface potential.
cdi_status cdi_psi_coupled(cdi_domain *d) {
  CDI_TRY(d, cudaMemsetAsync(d->d_src, 0, (size_t)d->N * 8, d->stream), "charge reset");
  const double F = 96485.0, eps0 = 8.854e-12;
  const double coef = F * d->dx * d->dx / (d->eps_r * eps0);
  const int4 z = make_int4(d->z[0], d->z[1], d->z[2], d->z[3]);
  if (d->prec == CDI_FP64)
    k_charge<double><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        (int)d->n_pore, d->ns, d->d_cell_list, c_views<double>(d, d->d_C[d->cur]), z, coef,
        d->d_src);
  else
    k_charge<float><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        (int)d->n_pore, d->ns, d->d_cell_list, c_views<float>(d, d->d_C[d->cur]), z, coef,
        d->d_src);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "charge");
  int it = 0;
  double rel = 0.0;
  // converged or not, the solve replaces the potential that both schemes'
  // face coefficients were formed from
  d->faces_stale = d->imp_stale = true;
  cdi_status s = cdi_psi_solve(d, d->psi_s, 0.0, d->d_src, d->psi_tol, d->psi_max_iter, &it, &rel);
  if (s == CDI_ERR_NOT_CONVERGED)
    return cdi_fail(d, s, "coupled potential did not reach tol within max_iter");
  return s;
}
