// Implicit (backward Euler) finite-volume transport: the time integration
// Sec. 2 uses for Eq. 3 with the adsorption flux of Eq. 6.  Each step solves,
// per species,
//   (I + dt A) C^{n+1} = C^n + dt b,
// where (1/dx) sum_f J_f(C) = A C - b are the face fluxes of the explicit
// step (Scharfetter-Gummel fluxes with frozen velocity and potential, the
// half-cell Robin closure at solid faces, the feed ghost at the inlet, the
// copying ghost at the outlet).  The operator is assembled once per
// transport state in FP64 (a diagonal, one coefficient per face and the
// account coefficients, by pore rank); the solve is matrix-free, Jacobi-
// preconditioned BiCGStab in FP64, all of it in one cooperative launch with
// fixed-order sums, so a run is deterministic.  The adsorbed,
// inflow and outflow accounts take the fluxes at C^{n+1}, so the mass balance
// closes as in the explicit scheme.  The step is unconditionally stable and
// positivity-preserving (I + dt A is an M-matrix), so dt may exceed the
// explicit bound by orders of magnitude.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "cdi_internal.cuh"

using namespace cdi;

namespace {

// Scalar slots of the solver (d_iscal): per species of a launch its last
// relative residual and iterations, then the launch's verdict (0: every
// species converged) and the barrier's (0: no barrier ran into its limit).
enum { B_REL = 0, B_IT = kMaxSpecies, B_FAIL = 2 * kMaxSpecies, B_BAR, B_N };

// The solver works on y = K x, K = 1 + dt A_PP (Jacobi preconditioning from
// the right), so that an iteration has neither divisions nor the diagonal:
// M y = y_P + sum_f off_f y_nb with off_f = dt a_f / K_nb formed once per
// operator.  At 2 FP64 operations a clock and SM the arithmetic bounds an
// iteration; a division is worth about ten multiply-adds.
//
// Coefficients of species k, component j at ((k * NC) + j) * n + r: K, off of
// the faces (+x, -x, +y, -y, +z, -z; exactly 0 across a closed face), and
// the account coefficients ain = (D/dx) B(-P_in), bin = (D/dx) B(P_in) c0
// (the inflow is bin - ain C_P), aout = (D/dx) (B(-P_out) - B(P_out))
// (outflow aout C_P).
template <int DIM> struct ICoef {
  static constexpr int NF = 2 * DIM;
  static constexpr int K = 0, FACE = 1, AIN = 1 + NF, BIN = 2 + NF, AOUT = 3 + NF, NC = 4 + NF;
};
constexpr int kImpVecs = 5;  // r, r0, p, v, t per species

struct IGeo {
  const NFlag *fl;   // per rank face flags
  const int *lat;    // lateral neighbour ranks (-1: none)
  int n, walls;
};

// Neighbour rank across face fc of rank r (-1: none) and the face kind.
enum { K_PORE = 0, K_SOLID = 1, K_INLET = 2, K_OUTLET = 3, K_WALL = 4 };
__device__ __forceinline__ int ikind(const IGeo &g, unsigned f, int fc, int r, int &q) {
  const bool solid = (f >> (kFaceBit + fc)) & 1u;
  const bool edge = (f >> (kEdgeBit + fc)) & 1u;
  q = -1;
  if (fc < 2) {
    if (edge) return fc == 0 ? K_OUTLET : K_INLET;
    if (solid) return K_SOLID;
    q = r + (fc == 0 ? 1 : -1);
    return K_PORE;
  }
  if (edge && g.walls) return K_WALL;
  if (solid) return K_SOLID;
  q = g.lat[(size_t)(fc - 2) * g.n + r];
  return q >= 0 ? K_PORE : K_SOLID;
}

__device__ __forceinline__ double phi_of(double v) { return v; }
__device__ __forceinline__ double phi_of(float2 v) { return (double)v.x + (double)v.y; }

// Per-species constants passed by value.
struct PerSpecies {
  double v[kMaxSpecies];
};

template <typename T, int DIM>
__global__ void k_imp_coef(IGeo g, const T *__restrict__ u,
                           const typename PhiStore<T>::type *__restrict__ phi, int ns,
                           PerSpecies dxD, PerSpecies Ddx, PerSpecies Keff, PerSpecies zf,
                           double inv_dx, double c0, double dt, double *__restrict__ co) {
  using C = ICoef<DIM>;
  const double *dxDk = dxD.v, *Ddxk = Ddx.v, *Kk = Keff.v, *zk = zf.v;
  const size_t n = (size_t)g.n;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < g.n; r += gridDim.x * blockDim.x) {
    const unsigned f = g.fl[r];
    const double phP = phi_of(phi[r]);
    for (int k = 0; k < ns; k++) {
      double *c = co + (size_t)k * C::NC * n;
      double diag = 0.0, ain = 0.0, bin = 0.0, aout = 0.0;
      for (int fc = 0; fc < C::NF; fc++) {
        int q;
        const int kind = ikind(g, f, fc, r, q);
        double off = 0.0;
        if (kind == K_SOLID) {
          diag += Kk[k] * inv_dx;
        } else if (kind != K_WALL) {
          const int a = fc >> 1;
          const double uP = (double)u[(size_t)a * n + r];
          const double un = kind == K_PORE ? (double)u[(size_t)a * n + q] : uP;
          const double phn = kind == K_PORE ? phi_of(phi[q]) : (kind == K_INLET ? 0.0 : phP);
          const double half = (fc & 1) ? -0.5 : 0.5;
          const double P = half * (uP + un) * dxDk[k] - zk[k] * (phn - phP);
          double Bp, Bm;
          bernoulli_pair(P, Bp, Bm);
          if (kind == K_PORE) {
            diag += Ddxk[k] * inv_dx * Bm;
            off = -Ddxk[k] * inv_dx * Bp;
          } else if (kind == K_INLET) {
            diag += Ddxk[k] * inv_dx * Bm;
            ain = Ddxk[k] * Bm;
            bin = Ddxk[k] * Bp * c0;
          } else {
            diag += Ddxk[k] * inv_dx * (Bm - Bp);
            aout = Ddxk[k] * (Bm - Bp);
          }
        }
        c[(size_t)(C::FACE + fc) * n + r] = off;
      }
      c[(size_t)C::K * n + r] = 1.0 + dt * diag;
      c[(size_t)C::AIN * n + r] = ain;
      c[(size_t)C::BIN * n + r] = bin;
      c[(size_t)C::AOUT * n + r] = aout;
    }
  }
}

// off_f = dt a_f / K_nb, once every K stands.
template <int DIM>
__global__ void k_imp_scale(IGeo g, int ns, double dt, double *__restrict__ co) {
  using C = ICoef<DIM>;
  const size_t n = (size_t)g.n;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < g.n; r += gridDim.x * blockDim.x) {
    const unsigned f = g.fl[r];
    for (int fc = 0; fc < C::NF; fc++) {
      int q;
      if (ikind(g, f, fc, r, q) != K_PORE) continue;
      for (int k = 0; k < ns; k++) {
        double *c = co + (size_t)k * C::NC * n;
        double *o = c + (size_t)(C::FACE + fc) * n + r;
        *o = dt * *o / c[(size_t)C::K * n + q];
      }
    }
  }
}

// The neighbours of rank r across its open faces: fn(q, off) in face order.
// A closed face has off exactly +0 (an integer test: an FP64 comparison would
// take the FP64 pipe); its q is not formed.
template <int DIM, typename F>
__device__ __forceinline__ void open_faces(const int *__restrict__ lat,
                                           const double *__restrict__ off, size_t n, int r, F fn) {
  double o[2 * DIM];
  int q[2 * DIM];
#pragma unroll
  for (int f = 0; f < 2 * DIM; f++) {
    o[f] = off[(size_t)f * n + r];
    q[f] = f < 2 ? r + (f == 0 ? 1 : -1) : lat[(size_t)(f - 2) * n + r];
  }
#pragma unroll
  for (int f = 0; f < 2 * DIM; f++)
    if (__double_as_longlong(o[f]) != 0) fn(q[f], o[f]);
}

template <typename T> struct BiArgs {
  const double *co;   // coefficients of the launch's first species
  const int *lat;
  int n, ns, max_iter;
  double dt_dx, tol;  // dt / dx
  CViews<T> C;        // C^n of the launch's species
  double *y;          // a vector per species, the solution
  double *w;          // kImpVecs vectors per species
  double *part, *scal;
  unsigned *counter;
};

// One backward Euler step's linear solves, all species of the launch side by
// side: Jacobi-preconditioned BiCGStab from the first guess C^n, the
// iterations and their dot products in one cooperative launch.
//
// What bounds it: FP64 arithmetic (31 operations a cell, species and
// iteration in 3D), then the four grid barriers of an iteration.  Before, an
// iteration was four launches a species, divided by K of every neighbour in
// both products and summed by five FP64 shuffle rounds a warp: 80^3, two
// species, 6 steps of 40 explicit ones 40.5 -> 11.1 ms.  The neighbours'
// s = r - alpha v are formed on the fly: a pass of their own would cost
// another barrier.
template <typename T, int DIM>
__global__ void __launch_bounds__(kGridThreads) k_bi_solve(BiArgs<T> a) {
  using C = ICoef<DIM>;
  extern __shared__ double sm[];  // 2 ns rows of a value a thread (GridBarrier)
  __shared__ double tot[kGridSums];
  __shared__ double rho[kMaxSpecies], alpha[kMaxSpecies], omega[kMaxSpecies], beta[kMaxSpecies],
      bb[kMaxSpecies], rr2[kMaxSpecies], limit[kMaxSpecies];
  __shared__ int it[kMaxSpecies], done[kMaxSpecies];
  const size_t n = (size_t)a.n;
  const int first = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  GridBarrier bar{a.counter, a.part, sm, (int)blockDim.x, 0u, 0};

  for (int k = 0; k < a.ns; k++) {
    const double *c = a.co + (size_t)k * C::NC * n;
    double *y = a.y + (size_t)k * n;
    double *rr = a.w + (size_t)k * kImpVecs * n, *r0 = rr + n, *p = r0 + n;
    const CView<T> Ck = a.C.v[k];
    double v[2] = {0.0, 0.0};
    for (int r = first; r < a.n; r += stride) {
      const double cP = Ck.at(r), yP = c[(size_t)C::K * n + r] * cP;
      const double rhs = cP + a.dt_dx * c[(size_t)C::BIN * n + r];
      double My = yP;
      open_faces<DIM>(a.lat, c + (size_t)C::FACE * n, n, r,
                      [&](int q, double o) { My += o * (c[(size_t)C::K * n + q] * Ck.at(q)); });
      const double res = rhs - My;
      y[r] = yP;
      rr[r] = res;
      r0[r] = res;
      p[r] = res;
      v[0] += res * res;
      v[1] += rhs * rhs;
    }
    grid_add(bar, 2 * k, v[0]);
    grid_add(bar, 2 * k + 1, v[1]);
  }
  if (!grid_totals(bar, tot, 2 * a.ns)) return grid_give_up(a.scal + B_BAR);
  if (threadIdx.x < a.ns) {
    const int k = threadIdx.x;
    rho[k] = tot[2 * k];
    bb[k] = tot[2 * k + 1];
    rr2[k] = rho[k];
    limit[k] = a.tol * a.tol * bb[k];  // of r . r
    it[k] = 0;
    done[k] = rr2[k] < limit[k] || bb[k] == 0.0 || rho[k] == 0.0;
  }
  __syncthreads();

  for (int step = 0; step < a.max_iter; step++) {
    bool all = true;
    for (int k = 0; k < a.ns; k++) all = all && done[k];
    if (all) break;

    // v = M p; alpha = rho / (r0 . v)
    for (int k = 0; k < a.ns; k++) {
      double v[1] = {0.0};
      if (!done[k]) {
        const double *off = a.co + ((size_t)k * C::NC + C::FACE) * n;
        double *rr = a.w + (size_t)k * kImpVecs * n, *vv = rr + 3 * n;
        const double *r0 = rr + n, *p = rr + 2 * n;
        for (int r = first; r < a.n; r += stride) {
          double m = p[r];
          open_faces<DIM>(a.lat, off, n, r, [&](int q, double o) { m += o * p[q]; });
          vv[r] = m;
          v[0] += r0[r] * m;
        }
      }
      grid_add(bar, k, v[0]);
    }
    if (!grid_totals(bar, tot, a.ns)) return grid_give_up(a.scal + B_BAR);
    if (threadIdx.x < a.ns && !done[threadIdx.x])
      alpha[threadIdx.x] = tot[threadIdx.x] != 0.0 ? rho[threadIdx.x] / tot[threadIdx.x] : 0.0;
    __syncthreads();

    // s = r - alpha v, t = M s; omega = (t . s) / (t . t)
    for (int k = 0; k < a.ns; k++) {
      double v[2] = {0.0, 0.0};
      if (!done[k]) {
        const double *off = a.co + ((size_t)k * C::NC + C::FACE) * n;
        double *t = a.w + ((size_t)k * kImpVecs + 4) * n;
        const double *rr = t - 4 * n, *vv = t - n;
        const double al = alpha[k];
        for (int r = first; r < a.n; r += stride) {
          const double sP = rr[r] - al * vv[r];
          double m = sP;
          open_faces<DIM>(a.lat, off, n, r,
                          [&](int q, double o) { m += o * (rr[q] - al * vv[q]); });
          t[r] = m;
          v[0] += m * sP;
          v[1] += m * m;
        }
      }
      grid_add(bar, 2 * k, v[0]);
      grid_add(bar, 2 * k + 1, v[1]);
    }
    if (!grid_totals(bar, tot, 2 * a.ns)) return grid_give_up(a.scal + B_BAR);
    if (threadIdx.x < a.ns && !done[threadIdx.x]) {
      const int k = threadIdx.x;
      omega[k] = tot[2 * k + 1] != 0.0 ? tot[2 * k] / tot[2 * k + 1] : 0.0;
    }
    __syncthreads();

    // y += alpha p + omega s, r = s - omega t; rho' = r0 . r
    for (int k = 0; k < a.ns; k++) {
      double v[2] = {0.0, 0.0};
      if (!done[k]) {
        double *y = a.y + (size_t)k * n, *rr = a.w + (size_t)k * kImpVecs * n;
        const double *r0 = rr + n, *p = rr + 2 * n, *vv = rr + 3 * n, *t = rr + 4 * n;
        const double al = alpha[k], om = omega[k];
        for (int r = first; r < a.n; r += stride) {
          const double sP = rr[r] - al * vv[r];
          y[r] += al * p[r] + om * sP;
          const double rv = sP - om * t[r];
          rr[r] = rv;
          v[0] += r0[r] * rv;
          v[1] += rv * rv;
        }
      }
      grid_add(bar, 2 * k, v[0]);
      grid_add(bar, 2 * k + 1, v[1]);
    }
    if (!grid_totals(bar, tot, 2 * a.ns)) return grid_give_up(a.scal + B_BAR);
    if (threadIdx.x < a.ns && !done[threadIdx.x]) {
      const int k = threadIdx.x;
      const double r1 = tot[2 * k];
      // one division: a chain of FP64 latencies that all threads wait for
      const double div = rho[k] * omega[k];
      beta[k] = div != 0.0 ? r1 * alpha[k] / div : 0.0;
      rho[k] = r1;
      rr2[k] = tot[2 * k + 1];
      it[k]++;
      // converged, or broken down (no new direction)
      if (rr2[k] < limit[k] || bb[k] == 0.0 || r1 == 0.0 || omega[k] == 0.0) done[k] = 1;
    }
    __syncthreads();

    // p = r + beta (p - omega v)
    for (int k = 0; k < a.ns; k++) {
      if (done[k]) continue;
      double *p = a.w + ((size_t)k * kImpVecs + 2) * n;
      const double *rr = p - 2 * n, *vv = p + n;
      const double be = beta[k], om = omega[k];
      for (int r = first; r < a.n; r += stride) p[r] = rr[r] + be * (p[r] - om * vv[r]);
    }
    if (!grid_totals(bar, tot, 0)) return grid_give_up(a.scal + B_BAR);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    for (int k = 0; k < a.ns; k++) {
      const double rel = bb[k] > 0.0 ? sqrt(rr2[k] / bb[k]) : 0.0;
      a.scal[B_REL + k] = rel;
      a.scal[B_IT + k] = it[k];
      if (!(rr2[k] < limit[k] || rel < a.tol)) a.scal[B_FAIL] = 1.0;
    }
  }
}

// C^{n+1} = y / K into the storage type (an FP32 pair splits into hi + lo),
// unless a solve of the step failed (the step is then not taken), and the
// accounts of the step: the adsorbed, inflow and outflow fluxes at
// C^{n+1}, summed per warp of 32 ranks into the domain's per-warp accounts.
template <typename T, int DIM>
__global__ void k_bi_finish(IGeo g, const double *__restrict__ c, const double *__restrict__ y,
                            const double *__restrict__ scal, double Keff, CView<T> Cout, int k,
                            typename std::conditional<std::is_same<T, float>::value, float2,
                                                      double>::type *__restrict__ acc,
                            int naccs) {
  using C = ICoef<DIM>;
  if (scal[B_FAIL] != 0.0 || scal[B_BAR] != 0.0) return;
  const size_t n = (size_t)g.n;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  double v[3] = {0.0, 0.0, 0.0};
  if (r < g.n) {
    const double xv = y[r] / c[(size_t)C::K * n + r];
    T *o = const_cast<T *>(Cout.p) + (size_t)r * Cout.stride;
    const T hi = (T)xv;
    o[0] = hi;
    if (Cout.lo) o[Cout.lo] = (T)(xv - (double)hi);
    const unsigned f = g.fl[r];
    int solids = 0, q;
    for (int fc = 0; fc < C::NF; fc++) solids += ikind(g, f, fc, r, q) == K_SOLID;
    v[0] = solids * Keff * xv;
    v[1] = c[(size_t)C::BIN * n + r] - c[(size_t)C::AIN * n + r] * xv;
    v[2] = c[(size_t)C::AOUT * n + r] * xv;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int j = 0; j < 3; j++) v[j] += __shfl_down_sync(0xffffffffu, v[j], o);
  const int w = r >> 5;
  if ((threadIdx.x & 31) == 0 && w < naccs) {
    for (int j = 0; j < 3; j++) {
      auto *a = acc + (size_t)(3 * k + j) * naccs + w;
      if constexpr (std::is_same<T, float>::value) {
        // an FP32 pair account: add the FP64 value as hi + lo, each by two-sum
        const float parts[2] = {(float)v[j], (float)(v[j] - (double)(float)v[j])};
        for (float pv : parts) {
          float2 tt = *a;
          const float sum = __fadd_rn(tt.x, pv);
          const float bp = __fsub_rn(sum, tt.x);
          const float e = __fadd_rn(__fsub_rn(tt.x, __fsub_rn(sum, bp)), __fsub_rn(pv, bp));
          tt.x = sum;
          tt.y = __fadd_rn(tt.y, e);
          *a = tt;
        }
      } else {
        *a = __dadd_rn(*a, v[j]);
      }
    }
  }
}

IGeo make_igeo(const cdi_domain *d) {
  return IGeo{d->d_cfl, d->d_latnb, (int)d->n_pore, d->walls};
}

template <typename T, int DIM>
cdi_status imp_coefs(cdi_domain *d) {
  PerSpecies dxD, Ddx, Keff, zf;
  for (int k = 0; k < kMaxSpecies; k++) {
    const double Dk = k < d->ns ? d->D[k] : 1.0;
    dxD.v[k] = d->dx / Dk;
    Ddx.v[k] = Dk / d->dx;
    Keff.v[k] = d->Ka / (1.0 + d->Ka * d->dx / (2.0 * Dk));
    zf.v[k] = k < d->ns ? d->z[k] : 0.0;
  }
  k_imp_coef<T, DIM><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
      make_igeo(d), (const T *)d->d_u, (const typename PhiStore<T>::type *)d->d_phi, d->ns,
      dxD, Ddx, Keff, zf, 1.0 / d->dx, d->c0, d->dt, d->d_icoef);
  k_imp_scale<DIM><<<kRedBlocks, kRedThreads, 0, d->stream>>>(make_igeo(d), d->ns, d->dt,
                                                              d->d_icoef);
  d->timing.kernel_launches += 2;
  CDI_TRY(d, cudaGetLastError(), "implicit operator");
  d->imp_stale = false;
  return CDI_OK;
}

// The solver's launch: the same for every step of a call.
struct BiShape {
  int side, blocks, threads;  // species side by side, and the grid
  size_t smem;
};

// One step: the species solved side by side in one launch where their vectors
// could be had, else one after the other in one set of vectors.  The solutions
// stand in the potential solver's scratch (kMaxSpecies doubles a cell) and are
// taken into the state and the accounts once every species has converged.
template <typename T, int DIM>
cdi_status imp_step(cdi_domain *d, const BiShape &shape) {
  using C = ICoef<DIM>;
  using A = typename std::conditional<std::is_same<T, float>::value, float2, double>::type;
  const int n = (int)d->n_pore;
  const size_t nn = (size_t)n;
  const IGeo g = make_igeo(d);
  const int in = d->cur;
  const int side = shape.side;
  CDI_TRY(d, cudaMemsetAsync(d->d_iscal, 0, B_N * sizeof(double), d->stream), "implicit scalars");
  for (int k0 = 0; k0 < d->ns; k0 += side) {
    BiArgs<T> a;
    a.co = d->d_icoef + (size_t)k0 * C::NC * nn;
    a.lat = d->d_latnb;
    a.n = n;
    a.ns = std::min(side, d->ns - k0);
    a.max_iter = d->imp_max_iter;
    a.dt_dx = d->dt / d->dx;
    a.tol = d->imp_tol;
    for (int k = 0; k < a.ns; k++) a.C.v[k] = c_view<T>(d, d->d_C[in], k0 + k);
    a.y = d->d_cg + (size_t)k0 * nn;
    a.w = d->d_iwork;
    a.part = d->d_part;
    a.scal = d->d_iscal;
    a.counter = d->d_counter + C_IMP;
    CDI_TRY(d, cudaMemsetAsync(a.counter, 0, sizeof(unsigned), d->stream), "implicit barrier");
    void *args[] = {&a};
    CDI_TRY(d, cudaLaunchCooperativeKernel((const void *)k_bi_solve<T, DIM>, dim3(shape.blocks),
                                           dim3(shape.threads), args, shape.smem, d->stream),
            "implicit solve");
    d->timing.kernel_launches++;
    const bool last = k0 + side >= d->ns;
    for (int k = 0; last && k < d->ns; k++) {
      const double Keff = d->Ka / (1.0 + d->Ka * d->dx / (2.0 * d->D[k]));
      k_bi_finish<T, DIM><<<(n + 127) / 128, 128, 0, d->stream>>>(
          g, d->d_icoef + (size_t)k * C::NC * nn, d->d_cg + (size_t)k * nn, d->d_iscal, Keff,
          c_view<T>(d, d->d_C[1 - in], k), k, (A *)d->d_acc, d->np_accs);
      d->timing.kernel_launches++;
    }
    CDI_TRY(d, cudaGetLastError(), "implicit step");
    CDI_TRY(d, cudaMemcpyAsync(d->h_scal + S_IMP, d->d_iscal, B_N * sizeof(double),
                               cudaMemcpyDeviceToHost, d->stream),
            "implicit result");
    CDI_TRY(d, cudaStreamSynchronize(d->stream), "implicit step");
    const double *h = d->h_scal + S_IMP;
    if (h[B_BAR] != 0.0) {
      // blocks may have left at different points
      return cdi_fail(d, CDI_ERR_CUDA, "implicit step: a grid barrier ran into its limit");
    }
    for (int k = 0; k < a.ns; k++) {
      d->imp_iters += (int64_t)h[B_IT + k];
      d->imp_last_rel = h[B_REL + k];
    }
    if (h[B_FAIL] != 0.0)
      return cdi_fail(d, CDI_ERR_NOT_CONVERGED,
                      "implicit step: the linear solve did not reach tol within max_iter");
  }
  d->cur = 1 - in;
  return CDI_OK;
}

template <typename T, int DIM>
cdi_status imp_steps(cdi_domain *d, int64_t n) {
  if (d->imp_stale) {
    cdi_status s = imp_coefs<T, DIM>(d);
    if (s != CDI_OK) return s;
  }
  // vectors for all species at once, where memory allows (the one set of
  // cdi_imp_prepare may have been given back)
  for (int sets : {d->ns, 1}) {
    if (d->imp_sets >= sets) continue;
    double *w = (double *)(sets > 1 ? cdi_dev_alloc : cdi_dev_need)(
        d, (size_t)sets * kImpVecs * d->n_pore * 8);
    if (!w) continue;
    cdi_dev_release(d, d->d_iwork);
    d->d_iwork = w;
    d->imp_sets = sets;
  }
  if (d->imp_sets < 1) return cdi_fail(d, CDI_ERR_OOM, "implicit scheme: device memory");
  BiShape shape;
  shape.side = std::min(d->ns, d->imp_sets);
  shape.blocks = grid_shape((const void *)k_bi_solve<T, DIM>, d->n_pore, 1, 2 * shape.side,
                            &shape.threads, &shape.smem);
  if (shape.blocks == 0) return cdi_fail(d, CDI_ERR_CUDA, "implicit step: no resident block");
  cudaEvent_t ev;
  cdi_timing_begin(d, &ev);
  for (int64_t i = 0; i < n; i++) {
    cdi_status s = imp_step<T, DIM>(d, shape);
    if (s != CDI_OK) {
      cdi_timing_end(d, ev, PH_NP, i);
      return s;
    }
    d->np_steps++;
  }
  cdi_timing_end(d, ev, PH_NP, n);
  return CDI_OK;
}

}  // namespace

// Work memory of the implicit scheme (allocated on first use, kept for the
// domain's life): the operator of every species and the vectors of one (the
// first step takes those of the others).
cdi_status cdi_imp_prepare(cdi_domain *d) {
  const int NC = d->dim == 2 ? ICoef<2>::NC : ICoef<3>::NC;
  if (!d->d_icoef) {  // all of it, or nothing
    void *p[3] = {cdi_dev_need(d, (size_t)kMaxSpecies * NC * d->n_pore * 8),
                  cdi_dev_need(d, (size_t)kImpVecs * d->n_pore * 8), cdi_dev_need(d, 16 * 8)};
    if (!p[0] || !p[1] || !p[2]) {
      for (void *q : p)
        if (q) cdi_dev_release(d, q);
      return cdi_fail(d, CDI_ERR_OOM, "implicit scheme: device memory");
    }
    d->d_icoef = (double *)p[0];
    d->d_iwork = (double *)p[1];
    d->d_iscal = (double *)p[2];
    d->imp_sets = 1;
    CDI_TRY(d, cudaMemsetAsync(d->d_iscal, 0, 16 * 8, d->stream), "implicit scalars");
  }
  d->imp_stale = true;
  return CDI_OK;
}

cdi_status cdi_imp_steps(cdi_domain *d, int64_t n) {
  if (d->prec == CDI_FP64)
    return d->dim == 2 ? imp_steps<double, 2>(d, n) : imp_steps<double, 3>(d, n);
  return d->dim == 2 ? imp_steps<float, 2>(d, n) : imp_steps<float, 3>(d, n);
}
