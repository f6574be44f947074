// Explicit finite-volume Nernst-Planck transport (Eq. 3) with the adsorption
// flux of Eq. 6, and the transport queries.
//
// Per pore cell P, species k, face f with outward normal n:
//   pore or ghost neighbour:  P_f = (u_f . n) dx / D_k - z_k (phi_nb - phi_P)
//                             J   = (D_k/dx) [B(-P_f) C_P - B(P_f) C_nb]
//     evaluated for |P_f| < 1/2 as (D_k/dx) [E (C_P - C_nb) + (P_f/2)(C_P + C_nb)]
//     with the even series E = B(P) + P/2, and otherwise as the two products
//     (each accurate on its own; B(-P)(C_P - C_nb) + P C_nb would cancel
//     catastrophically for large |P|)
//   solid face (Eq. 6):       J   = K_eff C_P,  K_eff = Ka / (1 + Ka dx/(2 D_k))
//   lateral wall:             J   = 0
// with B(x) = x / (exp(x) - 1) (exponential fitting of advection and
// migration against diffusion), u_f the mean of the two cell velocities,
// phi = psi / V_T (kept to FP64 accuracy; the face difference is rounded to
// the storage precision only after subtraction).  The inlet ghost holds
// C = c0, phi = 0, u = u_P; the outlet ghost copies the cell (zero gradient).
// Update: C_P -= (dt/dx) sum_f J.  Fields are stored by pore rank (see
// NPGeo).  Adsorbed / inflow / outflow fluxes are summed per warp into
// per-warp accounts (FP64, or FP32 pairs in FP32 storage; a fixed warp ->
// cells map, so the totals are deterministic).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "cdi_internal.cuh"

using namespace cdi;

namespace {

enum { F_PORE = 0, F_SOLID = 1, F_INLET = 2, F_OUTLET = 3, F_WALL = 4 };

template <typename T> struct NPConst {
  T dxD[kMaxSpecies];   // dx / D_k
  T Ddx[kMaxSpecies];   // D_k / dx
  T Keff[kMaxSpecies];  // half-cell closure of Eq. 6
  T zf[kMaxSpecies];    // valence
  T dtdx;               // dt / dx
  T c0;                 // feed concentration
  T c0lo;               // its low word (c0 - (T)c0) for pair storage
};

template <int DIM>
__global__ void k_np_flags(const uint8_t *__restrict__ mask, NFlag *__restrict__ fl, int nx,
                           int ny, int nz, int walls) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= nx) return;
  const int y = blockIdx.y, z = blockIdx.z;
  const long long P = ((long long)z * ny + y) * nx + x;
  unsigned f = mask[P] ? 1u : 0u;
  for (int fc = 0; fc < 2 * DIM; fc++) {
    const int a = fc >> 1, s = (fc & 1) ? -1 : 1;
    int X = x, Y = y, Z = z;
    bool edge = false;
    if (a == 0) {
      X += s;
      edge = X < 0 || X >= nx;
    } else if (a == 1) {
      Y += s;
      edge = Y < 0 || Y >= ny;
      Y = (Y + ny) % ny;
    } else {
      Z += s;
      edge = Z < 0 || Z >= nz;
      Z = (Z + nz) % nz;
    }
    if (edge) f |= 1u << (kEdgeBit + fc);
    if ((a == 0 && edge) || (edge && walls)) continue;
    if (mask[((long long)Z * ny + Y) * nx + X]) f |= 1u << (kFaceBit + fc);
  }
  fl[P] = (NFlag)f;
}

// Face kind of face fc of pore cell P and, for a pore neighbour, its index Q,
// from the flag word alone (the edge bits carry the boundary position).
template <int DIM>
__device__ __forceinline__ int np_face(unsigned f, int fc, int nx, int ny, int nz, int walls,
                                       long long P, long long &Q) {
  const int a = fc >> 1, s = (fc & 1) ? -1 : 1;
  const bool edge = (f >> (kEdgeBit + fc)) & 1u;
  if (a == 0) {
    if (edge) return s > 0 ? F_OUTLET : F_INLET;
    if ((f >> (kFaceBit + fc)) & 1u) return F_SOLID;
    Q = P + s;
    return F_PORE;
  }
  if (edge && walls) return F_WALL;
  if ((f >> (kFaceBit + fc)) & 1u) return F_SOLID;
  const long long stride = a == 1 ? (long long)nx : (long long)nx * ny;
  const long long extent = a == 1 ? ny : nz;
  Q = P + (edge ? -s * (extent - 1) * stride : s * stride);
  return F_PORE;
}

// Pore rank of the pore lattice cell (x, row): the rank of the first pore
// cell of its 32-cell word plus the pore cells before it in that word.
__device__ __forceinline__ int rank_of(const uint2 *__restrict__ words, int W, int row, int x) {
  const uint2 t = __ldg(words + (size_t)row * W + (x >> 5));
  return (int)t.x + __popc(t.y & ((1u << (x & 31)) - 1u));
}

// Row of the lateral (y: a = 1, z: a = 2) neighbour across face fc; rows wrap
// periodically (a wall face is never asked).  row = z * ny + y.
__device__ __forceinline__ int lateral_row(unsigned f, int fc, int row, int ny, int nz) {
  const int s = (fc & 1) ? -1 : 1;
  const bool edge = (f >> (kEdgeBit + fc)) & 1u;
  const int step = (fc >> 1) == 1 ? 1 : ny;
  const int ext = (fc >> 1) == 1 ? ny : nz;
  return row + (edge ? -s * (ext - 1) * step : s * step);
}

// Face flux divided by D/dx: J' = B(-P) C_P - B(P) C_nb, for the face Peclet
// number P = adv - z (phi_nb - phi_P).
//
// FP32: phi and P are carried as unevaluated pairs (hi + lo) where it
// matters: an exponent |P| rounded to FP32 costs a relative error of about
// |P| * 6e-8 in each Boltzmann factor exp(P), which accumulates across an
// electric double layer.
//  * |P| < 1/2 (almost every face): with the even function
//      E(P) = B(P) + P/2 = (P/2) coth(P/2) = 1 + P^2/12 - P^4/720 + P^6/30240 - ...
//    (Bernoulli numbers; the next term is below 3.3e-9 here),
//      J' = E (C_P - C_nb) + (P/2) (C_P + C_nb),
//    a sum of two small, accurately rounded terms.
//  * otherwise: B at the high part of |P| from expm1, corrected to first
//    order in the low part with B'(x) = B(x) ((1 - B(x)) / x - 1), and
//    B(-a) = B(a) + a; J' = B(-P) C_P - B(P) C_nb, each product accurate.
__device__ __noinline__ void bernoulli_pair_split(float adv, float z, float2 nb, float2 pp,
                                                  float &Bp, float &Bm) {
  // phi_nb - phi_P as dhi + dlo (two-sum of the high parts plus the lows)
  const float d = __fsub_rn(nb.x, pp.x);
  const float bv = __fsub_rn(d, nb.x);
  const float e = __fadd_rn(__fsub_rn(nb.x, __fsub_rn(d, bv)), __fsub_rn(-pp.x, bv));
  const float dhi = d, dlo = __fadd_rn(e, __fsub_rn(nb.y, pp.y));
  // P = adv - z (dhi + dlo) as ph + pl
  const float zd = __fmul_rn(z, dhi);
  const float zde = __fmaf_rn(z, dhi, -zd);
  const float ph = __fsub_rn(adv, zd);
  const float bb = __fsub_rn(ph, adv);
  const float phe = __fadd_rn(__fsub_rn(adv, __fsub_rn(ph, bb)), __fsub_rn(-zd, bb));
  const float pl = __fsub_rn(__fsub_rn(phe, zde), __fmul_rn(z, dlo));
  const bool neg = ph < 0.f;
  const float ah = neg ? -ph : ph, al = neg ? -pl : pl;
  // B(a) = a e^-a / (1 - e^-a) is below 1e-33 beyond a = 80
  float Ba = ah > 80.f ? 0.f : __fdividef(ah, expm1f(ah));
  Ba = __fmaf_rn(__fmul_rn(Ba, al), __fsub_rn(__fdividef(__fsub_rn(1.f, Ba), ah), 1.f), Ba);
  const float Bma = __fadd_rn(__fadd_rn(Ba, ah), al);
  Bp = neg ? Bma : Ba;
  Bm = neg ? Ba : Bma;
}

__device__ __forceinline__ double phi_diff(double nb, double pp) { return __dsub_rn(nb, pp); }
__device__ __forceinline__ float phi_diff(float2 nb, float2 pp) {
  return __fadd_rn(__fsub_rn(nb.x, pp.x), __fsub_rn(nb.y, pp.y));
}

// Geometry of the compact transport layout handed to the FP64 step kernels.
struct NPGeo {
  const NFlag *fl;     // per rank: its face flags
  const int *lat;      // per lateral face f (y+, y-, z+, z-) and rank r, at
                       // (f - 2) * n + r: the pore neighbour's rank, or -1
  int n;
  int naccs;           // account sets (one per warp), the same for any launch shape
};

// FP32 storage: warps of 31 home cells.  Warp w holds ranks 31 w - 1 ..
// 31 w + 30 in lanes 0..31; lane 0 (the last home cell of warp w - 1) is a
// halo.  Each lane evaluates the flux through the +x face of its cell; when
// the -x neighbour of a cell is a pore cell it is the rank before it, i.e.
// the lane before it, so that face's flux is the previous lane's +x flux
// with its sign flipped (one shuffle).  Every x face is then evaluated once
// instead of twice, and every lane of the warp takes the same path.
constexpr int kHome = 31;

// The fields of one FP32 transport state, by value as kernel parameters (one
// launch, one state) or in a member table (fused sweeps and batches).  The
// concentrations of a species pair stand together, one record per rank
// (c0, c1, and with pair storage their low words: 16 bytes), so a cell or a
// neighbour is one load.
struct NPFields {
  const float *C[2];             // per species pair: records read
  float *Co[2];                  // records written
  const float2 *fd[3];           // per + face: face velocity, potential difference
  const short *latd;             // lateral differences (y+, y-[, z+, z-]) per rank
  const int *latb;               // their bases per tile of 31 ranks
  const int *lat;                // full lateral ranks (kLatWide cells only)
  const float *ux;               // x velocity (inlet cells only)
  const float2 *phi;             // psi / V_T as (hi, lo) (|P| >= 1/2 and inlet only)
  const NFlag *fl;               // face flags
  const float2 *bern;            // (B(P), B(-P)) of + face a, rank r, species k at
                                 // (a * n + r) * ns + k, and of the feed face at
                                 // a = dim; set where |P| >= 1/2
  float2 *acc;                   // per-warp accounts
};
__host__ __device__ constexpr long long np_warps(long long n) { return (n + kHome - 1) / kHome; }

// FP64 storage: one explicit step of species k at the pore cell of rank r.
// Writes the new concentration and returns the cell's adsorbed, inflow and
// outflow fluxes in v (io: it has an inlet or outlet face).  One thread per
// cell and species: the arithmetic is a chain of FP64 operations at a rate of
// 2 a clock and SM, so more, shorter threads are what hides it.
//
// The outlet ghost copies the cell (J = u_x C_P), the feed ghost has C = c0
// and phi = 0, a closed face has no flux, and the adsorption flux of the n_s
// solid faces, n_s K_eff C_P, is added once per cell.
//
// co: the stored face coefficients ((D/dx) B(P), (D/dx) B(-P)) of + face a at
// co[a * n + r], and of the feed face at a = DIM (k_np_coef64); a - face is
// the + face of the cell across it with the two exchanged.  They take the
// exponentials and divisions (about 60 FP64 operations a face) out of the
// step: 128x64 image, two species: 17.0 -> 4.1 us a step.  co null (no memory
// for them): every face is evaluated from the velocity and the potential.
template <int DIM, bool EARLY>
__device__ __forceinline__ bool np_cell(const double *Cin, double *Cout,
                                        const double2 *__restrict__ co,
                                        const double *__restrict__ u,
                                        const double *__restrict__ phi, const NPGeo &g,
                                        unsigned f, int r, const NPConst<double> &c, int k,
                                        double (&v)[3]) {
  constexpr int NF = 2 * DIM;
  const size_t n = (size_t)g.n;
  const bool inlet = (f >> (kEdgeBit + 1)) & 1u, outlet = (f >> kEdgeBit) & 1u;
  int q[NF];  // rank across the face (own rank at the inlet and outlet), -1 closed
  q[0] = (f >> kFaceBit) & 1u ? -1 : (outlet ? r : r + 1);
  q[1] = (f >> (kFaceBit + 1)) & 1u ? -1 : (inlet ? r : r - 1);
#pragma unroll
  for (int fc = 2; fc < NF; fc++) q[fc] = g.lat[(size_t)(fc - 2) * n + r];
  double Cn[NF], Bp[NF], Bm[NF];
#pragma unroll
  for (int fc = 0; fc < NF; fc++) {
    Bp[fc] = Bm[fc] = 0.0;
    if (q[fc] < 0) continue;
    if (co) {
      const bool feed = fc == 1 && inlet, flip = (fc & 1) && !feed;
      const double2 b = co[feed ? DIM * n + r : (fc >> 1) * n + (flip ? q[fc] : r)];
      Bp[fc] = flip ? b.y : b.x;
      Bm[fc] = flip ? b.x : b.y;
    } else {
      const double *ua = u + (fc >> 1) * n;
      const double uf = r_mul((fc & 1) ? -0.5 : 0.5, r_add(ua[r], ua[q[fc]]));
      const double dd = phi_diff(fc == 1 && inlet ? 0.0 : phi[q[fc]], phi[r]);
      bernoulli_pair(r_fma(-c.zf[k], dd, r_mul(uf, c.dxD[k])), Bp[fc], Bm[fc]);
      Bp[fc] = r_mul(c.Ddx[k], Bp[fc]);
      Bm[fc] = r_mul(c.Ddx[k], Bm[fc]);
    }
  }
  if (EARLY) {
    pdl_wait();  // the step before has written C
    pdl_launch();
  }
  const double CP = Cin[r];
#pragma unroll
  for (int fc = 0; fc < NF; fc++) Cn[fc] = q[fc] < 0 ? 0.0 : Cin[q[fc]];
  if (inlet) Cn[1] = c.c0;
  const double ns_solid = (double)__popc(f & (((1u << NF) - 1u) << kFaceBit));
  v[0] = r_mul(r_mul(ns_solid, c.Keff[k]), CP);
  double sumJ = v[0];
#pragma unroll
  for (int fc = 0; fc < NF; fc++) {
    const double J = r_fma(Bm[fc], CP, -r_mul(Bp[fc], Cn[fc]));
    sumJ = r_add(sumJ, J);
    if (fc == 1 && inlet) v[1] = -J;
    if (fc == 0 && outlet) v[2] = J;
  }
  Cout[r] = r_fma(-c.dtdx, sumJ, CP);
  return inlet || outlet;
}

// Per-warp account slot: FP64 for FP64 storage; for FP32 storage an
// unevaluated pair of FP32 words (hi + lo, about 48 significant bits) kept
// with the two-sum transformation, so the step issues no FP64 instruction
// (this part's FP64 rate is a small fraction of its FP32 rate).  Both are
// 8 bytes.
template <typename T> struct AccSlot { using type = double; };
template <> struct AccSlot<float> { using type = float2; };

__device__ __forceinline__ void acc_add(double *a, double v) { *a = __dadd_rn(*a, v); }
__device__ __forceinline__ void acc_add(float2 *a, float v) {
  float2 t = *a;
  const float s = __fadd_rn(t.x, v);
  const float bp = __fsub_rn(s, t.x);
  const float e = __fadd_rn(__fsub_rn(t.x, __fsub_rn(s, bp)), __fsub_rn(v, bp));
  t.x = s;
  t.y = __fadd_rn(t.y, e);
  *a = t;
}
__device__ __forceinline__ double acc_value(double a) { return a; }
__device__ __forceinline__ double acc_value(float2 a) { return (double)a.x + (double)a.y; }

// Warp sums of one species' fluxes v (FP64), added by lane 0 to the warp's own
// accounts acc[kind * nw + wid], kind 0 Gamma, 1 In, 2 Out (a fixed warp ->
// cells map, so the totals are deterministic).  A warp without inlet or
// outlet cells skips the In/Out sums (its values are 0).  All 32 lanes of the
// warp must call it.
__device__ __forceinline__ void np_account(double (&v)[3], bool io, double *__restrict__ acc,
                                           int wid, int nw) {
  const bool any_io = __any_sync(0xffffffffu, io);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v[0] = r_add(v[0], __shfl_down_sync(0xffffffffu, v[0], o));
  if (any_io) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int j = 1; j < 3; j++) v[j] = r_add(v[j], __shfl_down_sync(0xffffffffu, v[j], o));
  }
  if ((threadIdx.x & 31) == 0) {
    double *a = acc + wid;
    acc_add(a, v[0]);
    if (any_io) {
      acc_add(a + nw, v[1]);
      acc_add(a + 2 * (size_t)nw, v[2]);
    }
  }
}

// (t.x + t.y) + v as a renormalised FP32 pair (two-sum): acc_add without the
// memory access.
__device__ __forceinline__ float2 pair_add(float2 t, float v) {
  const float s = __fadd_rn(t.x, v);
  const float bp = __fsub_rn(s, t.x);
  const float e = __fadd_rn(__fsub_rn(t.x, __fsub_rn(s, bp)), __fsub_rn(v, bp));
  return make_float2(s, __fadd_rn(t.y, e));
}

// The FP32 warp accounts, two species at a time: lanes 0-15 carry species 2p
// and lanes 16-31 species 2p + 1 after the first exchange, so the pair's sums
// take 5 shuffles instead of 10 and end in lanes 0 and 16, which keep one
// account slot each.  The sums are those of np_account's shuffle tree (every
// addition has the same two operands), so the bits are too.  Each slot
// belongs to one warp tile: it is read before the tile's arithmetic
// (np_account_read), so its latency does not end the tile.  (The inflow and
// outflow slots, touched by the few warps at the inlet and outlet, are read
// at the end.)
template <int NS>
__device__ __forceinline__ void np_account_read(float2 (&a)[(NS + 1) / 2], const float2 *acc,
                                                int wid, int nw) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int p = 0; p < (NS + 1) / 2; p++) {
    const int k = 2 * p + (lane >> 4);
    if ((lane & 15) == 0 && k < NS) a[p] = acc[(size_t)(3 * k) * nw + wid];
  }
}
// v[p]: the lane's adsorbed fluxes of species (2p, 2p + 1).
template <int NS>
__device__ __forceinline__ void np_account_f32(const float2 (&v)[(NS + 1) / 2],
                                               const float2 (&a)[(NS + 1) / 2], float2 *acc,
                                               int wid, int nw) {
  const int lane = threadIdx.x & 31;
  const bool hi = lane >= 16;
#pragma unroll
  for (int p = 0; p < (NS + 1) / 2; p++) {
    const bool two = 2 * p + 1 < NS;
    float own = v[p].x, other = v[p].x;
    if (two) {
      own = hi ? v[p].y : v[p].x;
      other = hi ? v[p].x : v[p].y;
    }
    own = r_add(own, __shfl_xor_sync(0xffffffffu, other, 16));
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) own = r_add(own, __shfl_down_sync(0xffffffffu, own, o));
    const int k = 2 * p + (hi ? 1 : 0);
    if ((lane & 15) == 0 && k < NS) acc[(size_t)(3 * k) * nw + wid] = pair_add(a[p], own);
  }
}
// The inflow (kind 1) and outflow (kind 2) sums of a warp with inlet or
// outlet cells, as np_account forms them.
template <int NS>
__device__ __forceinline__ void np_account_io(float (&v)[2 * NS], float2 *acc, int wid, int nw) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < 2 * NS; k++) v[k] = r_add(v[k], __shfl_down_sync(0xffffffffu, v[k], o));
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int k = 0; k < NS; k++) {
      acc_add(acc + (size_t)(3 * k + 1) * nw + wid, v[k]);
      acc_add(acc + (size_t)(3 * k + 2) * nw + wid, v[NS + k]);
    }
}

// Two species per packed FP32x2 operation (each component rounded exactly as
// the scalar operation would be).
__device__ __forceinline__ float2 bc(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 pneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 psub(float2 a, float2 b) { return __fadd2_rn(a, pneg(b)); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Second species of pair p (a copy of the first when NS is odd).
template <int NS> __device__ __forceinline__ constexpr int np_k1(int p) {
  return 2 * p + 1 < NS ? 2 * p + 1 : 2 * p;
}

// The concentration record of rank r in a species-pair plane (two != 0: both
// species of the pair; else a lone last species, copied into both halves).
// Read through the non-coherent path, except behind a wait (EARLY: see
// pdl_wait).
template <bool EARLY, typename V> __device__ __forceinline__ V rec_get(const V *p) {
  if constexpr (EARLY) return *p;
  else return __ldg(p);
}
template <bool PAIR, bool EARLY>
__device__ __forceinline__ void rec_load(const float *base, bool two, int r, float2 &c,
                                         float2 &l) {
  if (PAIR && two) {
    const float4 v = rec_get<EARLY>(reinterpret_cast<const float4 *>(base) + r);
    c = make_float2(v.x, v.y);
    l = make_float2(v.z, v.w);
  } else if (two) {
    c = rec_get<EARLY>(reinterpret_cast<const float2 *>(base) + r);
    l = make_float2(0.f, 0.f);
  } else if (PAIR) {
    const float2 v = rec_get<EARLY>(reinterpret_cast<const float2 *>(base) + r);
    c = bc(v.x);
    l = bc(v.y);
  } else {
    c = bc(rec_get<EARLY>(base + r));
    l = make_float2(0.f, 0.f);
  }
}
template <bool PAIR>
__device__ __forceinline__ void rec_store(float *__restrict__ base, bool two, int r, float2 c,
                                          float2 l) {
  if (PAIR && two)
    reinterpret_cast<float4 *>(base)[r] = make_float4(c.x, c.y, l.x, l.y);
  else if (two)
    reinterpret_cast<float2 *>(base)[r] = c;
  else if (PAIR)
    reinterpret_cast<float2 *>(base)[r] = make_float2(c.x, l.x);
  else
    base[r] = c.x;
}

// Scalar flux of one species (pair-stored concentrations C + Cl with PAIR):
// the two branches above, the Bernoulli pair supplied by bern(Bp, Bm) where |P| >= 1/2;
// with PAIR the difference C_P - C_nb and the two products take the low words
// along.
template <bool PAIR, typename BF>
__device__ __forceinline__ float face_flux_one(float p, BF bern, float CP, float Cn, float CPl,
                                               float Cnl) {
  if (fabsf(p) < 0.5f) {
    const float p2 = __fmul_rn(p, p);
    float E = __fmaf_rn(p2, 1.f / 30240.f, -1.f / 720.f);
    E = __fmaf_rn(E, p2, 1.f / 12.f);
    E = __fmaf_rn(E, p2, 1.f);
    float dC = __fsub_rn(CP, Cn);
    if (PAIR) dC = __fadd_rn(dC, __fsub_rn(CPl, Cnl));
    return __fmaf_rn(E, dC, __fmul_rn(__fmul_rn(0.5f, p), __fadd_rn(CP, Cn)));
  }
  float Bp, Bm;
  bern(Bp, Bm);
  const float J = r_fma(Bm, CP, -r_mul(Bp, Cn));
  return PAIR ? __fadd_rn(J, r_fma(Bm, CPl, -r_mul(Bp, Cnl))) : J;
}

// Face Peclet numbers of a pair of species (k0, k1) from the face's velocity
// and potential difference seen from the cell.
__device__ __forceinline__ float2 face_peclet(float uf, float dd, const NPConst<float> &c, int k0,
                                              int k1) {
  return make_float2(__fmaf_rn(-c.zf[k0], dd, __fmul_rn(uf, c.dxD[k0])),
                     __fmaf_rn(-c.zf[k1], dd, __fmul_rn(uf, c.dxD[k1])));
}
__device__ __forceinline__ bool big(float2 p) { return !(fabsf(p.x) < 0.5f && fabsf(p.y) < 0.5f); }

// Flux through one face for a pair of species (k0, k1), times D/dx: for
// |P| < 1/2 both species at once in packed arithmetic, otherwise species by
// species (the same operations, each rounded the same way).  p: the face
// Peclet numbers; bern(k, Bp, Bm) supplies species k's Bernoulli pair and is
// asked only where |P| >= 1/2 (never with SMALL, whose caller knows that
// |P| < 1/2 for both).  An odd species count pads its last pair with a copy
// of the last species (k1 = k0).
template <bool PAIR, bool SMALL, typename BF>
__device__ __forceinline__ float2 face_flux_pair(float2 p, BF bern, float2 CP, float2 Cn,
                                                 float2 CPl, float2 Cnl, const NPConst<float> &c,
                                                 int k0, int k1) {
  float2 J;
  if (SMALL || !big(p)) {
    const float2 p2 = pmul(p, p);
    float2 E = pfma(p2, bc(1.f / 30240.f), bc(-1.f / 720.f));
    E = pfma(E, p2, bc(1.f / 12.f));
    E = pfma(E, p2, bc(1.f));
    float2 dC = psub(CP, Cn);
    if (PAIR) dC = padd(dC, psub(CPl, Cnl));
    J = pfma(E, dC, pmul(pmul(bc(0.5f), p), padd(CP, Cn)));
  } else {
    auto b0 = [&](float &Bp, float &Bm) { bern(k0, Bp, Bm); };
    auto b1 = [&](float &Bp, float &Bm) { bern(k1, Bp, Bm); };
    J.x = face_flux_one<PAIR>(p.x, b0, CP.x, Cn.x, CPl.x, Cnl.x);
    J.y = face_flux_one<PAIR>(p.y, b1, CP.y, Cn.y, CPl.y, Cnl.y);
  }
  return pmul(make_float2(c.Ddx[k0], c.Ddx[k1]), J);
}

// (s, e) with s + e = a + b exactly (two-sum, component-wise).
__device__ __forceinline__ void ptwo_sum(float2 a, float2 b, float2 &s, float2 &e) {
  s = padd(a, b);
  const float2 bp = psub(s, a);
  e = padd(psub(a, psub(s, bp)), psub(b, bp));
}

// The per-lane link data of warp w's tile: the lane's face flags (a lane
// without a cell has a closed +x face) and its lateral neighbour ranks (-1
// across a solid face or wall, or for the halo lane), decoded from the 16-bit
// differences to the tile's bases.
template <int DIM> struct NPLinks {
  unsigned f;
  int q[2 * DIM - 2];
};
template <int DIM>
__device__ __forceinline__ NPLinks<DIM> np_links(const NPFields &F, int n_cells, int w) {
  const int lane = threadIdx.x & 31;
  const int r = kHome * w + lane - 1;
  const bool valid = r >= 0 && r < n_cells;
  const bool home = valid && lane != 0;
  NPLinks<DIM> L;
  L.f = valid ? (unsigned)F.fl[r] : 1u << kFaceBit;
  int base[2 * DIM - 2], d[2 * DIM - 2];
  bool wide = false;
  if constexpr (DIM == 3) {
    const int4 b = reinterpret_cast<const int4 *>(F.latb)[w];
    short4 v = make_short4(kLatClosed, kLatClosed, kLatClosed, kLatClosed);
    if (home) v = reinterpret_cast<const short4 *>(F.latd)[r];
    base[0] = b.x; base[1] = b.y; base[2] = b.z; base[3] = b.w;
    d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
  } else {
    const int2 b = reinterpret_cast<const int2 *>(F.latb)[w];
    short2 v = make_short2(kLatClosed, kLatClosed);
    if (home) v = reinterpret_cast<const short2 *>(F.latd)[r];
    base[0] = b.x; base[1] = b.y;
    d[0] = v.x; d[1] = v.y;
  }
#pragma unroll
  for (int j = 0; j < 2 * DIM - 2; j++) {
    L.q[j] = d[j] == kLatClosed ? -1 : r + base[j] + d[j];
    wide |= d[j] == kLatWide;
  }
  if (wide) {
#pragma unroll
    for (int j = 0; j < 2 * DIM - 2; j++) L.q[j] = F.lat[(size_t)j * n_cells + r];
  }
  return L;
}

// What a lane works from: its cell's record, the records across its +x and
// lateral faces (its own again across a closed face) and the face data seen
// from the cell (0 across a closed face).
template <int DIM, int NS> struct NPLane {
  static constexpr int NP = (NS + 1) / 2, NL = 2 * DIM - 2;
  float2 C[NP], Cl[NP];
  float2 Cx[NP], Cxl[NP], fx;
  float2 Cn[NL][NP], Cnl[NL][NP], fn[NL];
};

// The update of warp w's tile from the values in V.  The +x face flux is
// evaluated once per face and handed to the next lane as its -x flux; per
// home cell the faces are summed in the order adsorption, +x, -x, +y,
// -y, +z, -z.  SMALL: every face of the warp has |P| < 1/2, so the
// arithmetic has no branch and its faces overlap.  EVAL: the Bernoulli pairs
// are not stored (no memory for them) and are evaluated at every step.
template <int DIM, int NS, bool PAIR, bool SMALL, bool EVAL>
__device__ __forceinline__ void np_update(const NPFields &F, int n_cells, int naccs,
                                          const NPConst<float> &c, int w, int r, bool home,
                                          const NPLinks<DIM> &lk, const NPLane<DIM, NS> &V,
                                          const float2 (&acc_pre)[(NS + 1) / 2]) {
  constexpr int NF = 2 * DIM, NL = NF - 2, NP = (NS + 1) / 2;
  const unsigned f = lk.f;
  const float2 z2 = make_float2(0.f, 0.f);
  const int rc = min(max(r, 0), n_cells - 1);
  const bool xs = (f >> kFaceBit) & 1u, xe = (f >> kEdgeBit) & 1u;
  const bool ms = (f >> (kFaceBit + 1)) & 1u, me = (f >> (kEdgeBit + 1)) & 1u;
  float2 Jx[NP], Jm[NP];
  // The Bernoulli pair of species k at + face a of rank own, or (flip) at the
  // - face of the cell across it: the stored pair, with its two members
  // exchanged there, or evaluated from the two potentials.
  auto stored = [&](int a, int own, bool flip, float uf, float dd, int nb, int k, float &Bp,
                    float &Bm) {
    if (!EVAL) {
      const float2 b = F.bern[((size_t)a * n_cells + own) * NS + k];
      Bp = flip ? b.y : b.x;
      Bm = flip ? b.x : b.y;
    } else {
      bernoulli_pair_split(__fmul_rn(uf, c.dxD[k]), c.zf[k], F.phi[nb], F.phi[rc], Bp, Bm);
    }
  };
#pragma unroll
  for (int p = 0; p < NP; p++) {
    auto bern = [&](int k, float &Bp, float &Bm) {
      stored(0, rc, false, V.fx.x, V.fx.y, xs || xe ? rc : rc + 1, k, Bp, Bm);
    };
    Jx[p] = face_flux_pair<PAIR, SMALL>(face_peclet(V.fx.x, V.fx.y, c, 2 * p, np_k1<NS>(p)), bern,
                                        V.C[p], V.Cx[p], V.Cl[p], V.Cxl[p], c, 2 * p,
                                        np_k1<NS>(p));
  }
  // -x face: the previous lane's +x face (pore neighbour), the feed ghost
  // (inlet), or closed (solid)
#pragma unroll
  for (int p = 0; p < NP; p++) {
    Jm[p].x = -__shfl_up_sync(0xffffffffu, Jx[p].x, 1);
    Jm[p].y = 2 * p + 1 < NS ? -__shfl_up_sync(0xffffffffu, Jx[p].y, 1) : Jm[p].x;
    if (ms) Jm[p] = z2;
  }
  if (home && me) {
    const float uP = F.ux[r];
    const float2 phP = F.phi[r];
    const float uf = r_mul(-0.5f, r_add(uP, uP));
    const float dd = phi_diff(z2, phP);
    auto bern = [&](int k, float &Bp, float &Bm) {
      if (!EVAL) {  // the feed faces' pairs stand behind those of the + faces
        const float2 b = F.bern[((size_t)DIM * n_cells + r) * NS + k];
        Bp = b.x;
        Bm = b.y;
      } else {
        bernoulli_pair_split(__fmul_rn(uf, c.dxD[k]), c.zf[k], z2, phP, Bp, Bm);
      }
    };
#pragma unroll
    for (int p = 0; p < NP; p++)
      Jm[p] = face_flux_pair<PAIR, SMALL>(face_peclet(uf, dd, c, 2 * p, np_k1<NS>(p)), bern, V.C[p],
                                          bc(c.c0), V.Cl[p], bc(c.c0lo), c, 2 * p,
                                          np_k1<NS>(p));
  }
  // adsorption on the solid faces (Eq. 6), then the faces in order
  float2 Ja[NP], sumJ[NP];
  const float ns_solid = (float)__popc(f & (((1u << NF) - 1u) << kFaceBit));
#pragma unroll
  for (int p = 0; p < NP; p++) {
    Ja[p] = pmul(pmul(bc(ns_solid), make_float2(c.Keff[2 * p], c.Keff[np_k1<NS>(p)])), V.C[p]);
    sumJ[p] = padd(padd(Ja[p], Jx[p]), Jm[p]);
  }
#pragma unroll
  for (int j = 0; j < NL; j++) {
    const int q = lk.q[j] >= 0 ? lk.q[j] : rc;
    auto bern = [&](int k, float &Bp, float &Bm) {
      stored(1 + j / 2, (j & 1) ? q : rc, j & 1, V.fn[j].x, V.fn[j].y, q, k, Bp, Bm);
    };
#pragma unroll
    for (int p = 0; p < NP; p++)
      sumJ[p] = padd(sumJ[p], face_flux_pair<PAIR, SMALL>(
                                  face_peclet(V.fn[j].x, V.fn[j].y, c, 2 * p, np_k1<NS>(p)), bern,
                                  V.C[p], V.Cn[j][p], V.Cl[p], V.Cnl[j][p], c, 2 * p,
                                  np_k1<NS>(p)));
  }
  if (home) {
#pragma unroll
    for (int p = 0; p < NP; p++) {
      float2 Cn, Cnl = z2;
      if (PAIR) {
        // (hi + lo) - dt/dx sum J by two-sum, renormalised
        float2 t, e;
        ptwo_sum(V.C[p], pmul(bc(-c.dtdx), sumJ[p]), t, e);
        const float2 l = padd(V.Cl[p], e);
        Cn = padd(t, l);
        Cnl = psub(l, psub(Cn, t));
      } else {
        Cn = pfma(bc(-c.dtdx), sumJ[p], V.C[p]);
      }
      rec_store<PAIR>(F.Co[p], 2 * p + 1 < NS, r, Cn, Cnl);
    }
  }
  if (!home) {
#pragma unroll
    for (int p = 0; p < NP; p++) Ja[p] = z2;
  }
  np_account_f32<NS>(Ja, acc_pre, F.acc, w, naccs);
  if (__any_sync(0xffffffffu, home && (me || xe))) {
    float v[2 * NS];
#pragma unroll
    for (int k = 0; k < NS; k++) {
      v[k] = home && me ? r_sub(0.f, (k & 1) ? Jm[k / 2].y : Jm[k / 2].x) : 0.f;
      v[NS + k] = home && xe ? r_add(0.f, (k & 1) ? Jx[k / 2].y : Jx[k / 2].x) : 0.f;
    }
    np_account_io<NS>(v, F.acc, w, naccs);
  }
}

// Every load of warp w's tile, the face data (which no step writes) before
// the wait for the step before.  All are unconditional: a closed face reads
// the cell's own record, which costs an L1 hit instead of a branch and moves.
template <int DIM, int NS, bool PAIR, bool EARLY>
__device__ __forceinline__ void np_load(const NPFields &F, int n_cells, int naccs, int w, int r,
                                        const NPLinks<DIM> &lk, NPLane<DIM, NS> &V,
                                        float2 (&acc_pre)[(NS + 1) / 2]) {
  constexpr int NL = 2 * DIM - 2, NP = (NS + 1) / 2;
  const int rc = min(max(r, 0), n_cells - 1);
  const bool xp = !(((lk.f >> kFaceBit) | (lk.f >> kEdgeBit)) & 1u);
  int q[NL];
#pragma unroll
  for (int j = 0; j < NL; j++) q[j] = lk.q[j] >= 0 ? lk.q[j] : rc;
  auto face = [&](int j) { V.fn[j] = __ldg(F.fd[1 + j / 2] + ((j & 1) ? q[j] : rc)); };
  if (EARLY) {
    V.fx = __ldg(F.fd[0] + rc);
#pragma unroll
    for (int j = 0; j < NL; j++) face(j);
    pdl_wait();
    pdl_launch();
  }
  np_account_read<NS>(acc_pre, F.acc, w, naccs);
#pragma unroll
  for (int p = 0; p < NP; p++) {
    rec_load<PAIR, EARLY>(F.C[p], 2 * p + 1 < NS, rc, V.C[p], V.Cl[p]);
    rec_load<PAIR, EARLY>(F.C[p], 2 * p + 1 < NS, xp ? rc + 1 : rc, V.Cx[p], V.Cxl[p]);
  }
  if (!EARLY) V.fx = __ldg(F.fd[0] + rc);
#pragma unroll
  for (int j = 0; j < NL; j++) {
#pragma unroll
    for (int p = 0; p < NP; p++)
      rec_load<PAIR, EARLY>(F.C[p], 2 * p + 1 < NS, q[j], V.Cn[j][p], V.Cnl[j][p]);
    if (!EARLY) face(j);
  }
#pragma unroll
  for (int j = 1; j < NL; j += 2) {
    // a - face is the + face of the neighbour across it, seen from the other
    // side: velocity and potential difference change sign exactly (and are 0
    // where it is closed)
    const float s = lk.q[j] >= 0 ? -1.f : 0.f;
    V.fn[j] = make_float2(__fmul_rn(s, V.fn[j].x), __fmul_rn(s, V.fn[j].y));
  }
}

// One explicit step of the home cells of warp w (FP32, NS species in
// (NS + 1) / 2 packed pairs), with the per-warp accounts of Gamma, In and
// Out.  PAIR: every concentration is an unevaluated pair hi + lo, updated
// with the two-sum transformation, so rounding does not build up over long
// runs; the fluxes take the low words into the concentration differences.
// All 32 lanes of the warp must call it.
//
// What bounds it is latency: a memory round trip for the link data, one for
// the gathers, and the arithmetic's own chain.  So every load is issued
// before any arithmetic, and the arithmetic of a launch whose faces all have
// |P| < 1/2 (NP_SMALL; known when the face data is formed) has no branch: a
// branch per face puts the faces' chains one after the other (172 instead of
// 139 us a step on a 256^3 pack), and even one vote per warp between the two
// costs the common one (150 to 172 us: the second path's registers).
// Otherwise (NP_LARGE) a vote per warp chooses; NP_EVAL is NP_LARGE without
// stored Bernoulli pairs.
enum { NP_SMALL = 0, NP_LARGE = 1, NP_EVAL = 2 };
template <int DIM, int NS, bool PAIR, int MODE, bool EARLY>
__device__ __forceinline__ void np_warp31(const NPFields &F, int n_cells, int naccs,
                                          const NPConst<float> &c, int w) {
  constexpr int NL = 2 * DIM - 2, NP = (NS + 1) / 2;
  constexpr bool EVAL = MODE == NP_EVAL;
  if (w >= (int)np_warps(n_cells)) return;  // whole warps
  const int r = kHome * w + (int)(threadIdx.x & 31) - 1;
  const bool valid = r >= 0 && r < n_cells, home = valid && (threadIdx.x & 31) != 0;
  const NPLinks<DIM> lk = np_links<DIM>(F, n_cells, w);
  NPLane<DIM, NS> V;
  float2 acc_pre[NP];
  np_load<DIM, NS, PAIR, EARLY>(F, n_cells, naccs, w, r, lk, V, acc_pre);
  if (MODE != NP_SMALL) {
    bool large = false;
#pragma unroll
    for (int p = 0; p < NP; p++) {
      large |= big(face_peclet(V.fx.x, V.fx.y, c, 2 * p, np_k1<NS>(p)));
#pragma unroll
      for (int j = 0; j < NL; j++)
        large |= big(face_peclet(V.fn[j].x, V.fn[j].y, c, 2 * p, np_k1<NS>(p)));
    }
    if (valid && ((lk.f >> (kEdgeBit + 1)) & 1u)) {  // the feed face
      const float uP = F.ux[r], uf = r_mul(-0.5f, r_add(uP, uP));
      const float dd = phi_diff(make_float2(0.f, 0.f), F.phi[r]);
#pragma unroll
      for (int p = 0; p < NP; p++) large |= big(face_peclet(uf, dd, c, 2 * p, np_k1<NS>(p)));
    }
    if (__any_sync(0xffffffffu, large)) {
      np_update<DIM, NS, PAIR, false, EVAL>(F, n_cells, naccs, c, w, r, home, lk, V, acc_pre);
      return;
    }
  }
  np_update<DIM, NS, PAIR, true, EVAL>(F, n_cells, naccs, c, w, r, home, lk, V, acc_pre);
}

// Rank across + face a of rank r (its own at the outlet), or -1 where closed.
__device__ __forceinline__ int plus_face(unsigned f, const int *__restrict__ lat, int n, int a,
                                         int r) {
  if (a > 0) return lat[(size_t)(2 * a - 2) * n + r];
  return (f >> kFaceBit) & 1u ? -1 : ((f >> kEdgeBit) & 1u ? r : r + 1);
}

// The face data of every + face, from the velocity and the potential: half
// the sum of the two cells' velocity components (the cell's own twice at the
// outlet) and the potential difference of the two (hi, lo) pairs, rounded
// once each; 0 across a closed face.  The step reads these 8 bytes instead
// of both cells' velocity and potential pair (12 bytes and three gathered
// loads per lateral face) and skips the arithmetic on them; they stay the
// same until the velocity or the potential changes.
// *any_large is set to 1 when a face has |P| >= 1/2 for some species.
template <int DIM>
__global__ void k_np_faces(const NFlag *__restrict__ fl, const int *__restrict__ lat, int n,
                           const float *__restrict__ u, const float2 *__restrict__ phi,
                           NPConst<float> c, int ns, float2 *__restrict__ fd,
                           int *__restrict__ any_large) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    const unsigned f = fl[r];
    const float2 phP = phi[r];
    bool large = false;
    auto test = [&](float uf, float dd) {
      for (int k = 0; k < ns; k++)
        if (!(fabsf(__fmaf_rn(-c.zf[k], dd, __fmul_rn(uf, c.dxD[k]))) < 0.5f)) large = true;
    };
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      const float uP = u[(size_t)a * n + r];
      const int q = plus_face(f, lat, n, a, r);
      float2 v = make_float2(0.f, 0.f);
      if (q >= 0) {
        v = make_float2(r_mul(0.5f, r_add(uP, u[(size_t)a * n + q])), phi_diff(phi[q], phP));
        test(v.x, v.y);
      }
      fd[(size_t)a * n + r] = v;
    }
    if ((f >> (kEdgeBit + 1)) & 1u)
      test(r_mul(-0.5f, r_add(u[r], u[r])), phi_diff(make_float2(0.f, 0.f), phP));
    if (large) *any_large = 1;
  }
}

// The Bernoulli pairs of the + faces and feed faces with |P| >= 1/2 (the
// others' places are not read): the step's exponentials and divisions, done
// once per velocity and potential instead of at every step.
template <int DIM>
__global__ void k_np_bern(const NFlag *__restrict__ fl, const int *__restrict__ lat, int n,
                          const float *__restrict__ ux, const float2 *__restrict__ phi,
                          const float2 *__restrict__ fd, NPConst<float> c, int ns,
                          float2 *__restrict__ bern) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    const unsigned f = fl[r];
    const float2 phP = phi[r];
    auto put = [&](int a, float uf, float dd, float2 nb) {
      for (int k = 0; k < ns; k++) {
        const float adv = __fmul_rn(uf, c.dxD[k]);
        if (fabsf(__fmaf_rn(-c.zf[k], dd, adv)) < 0.5f) continue;
        float Bp, Bm;
        bernoulli_pair_split(adv, c.zf[k], nb, phP, Bp, Bm);
        bern[((size_t)a * n + r) * ns + k] = make_float2(Bp, Bm);
      }
    };
    for (int a = 0; a < DIM; a++) {
      const int q = plus_face(f, lat, n, a, r);
      const float2 v = fd[(size_t)a * n + r];
      if (q >= 0) put(a, v.x, v.y, phi[q]);
    }
    if ((f >> (kEdgeBit + 1)) & 1u) {
      const float2 z2 = make_float2(0.f, 0.f);
      put(DIM, r_mul(-0.5f, r_add(ux[r], ux[r])), phi_diff(z2, phP), z2);
    }
  }
}

// 16-bit lateral differences of the tiles of 31 ranks (one warp per tile, as
// the step runs them): per face the tile's base is q - r of its first cell
// with an open face, and each cell keeps (q - r) - base, kLatClosed across a
// closed face, or kLatWide where it does not fit (the step then reads the
// full table).
template <int DIM>
__global__ void k_lat_pack(const int *__restrict__ lat, int n, short *__restrict__ latd,
                           int *__restrict__ latb) {
  constexpr int NL = 2 * DIM - 2;
  const int lane = threadIdx.x & 31;
  const int nw = (int)np_warps(n), W = gridDim.x * (blockDim.x >> 5);
  for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nw; w += W) {
    const int r = kHome * w + lane - 1;
    const bool home = lane != 0 && r < n;
#pragma unroll
    for (int j = 0; j < NL; j++) {
      const int q = home ? lat[(size_t)j * n + r] : -1;
      const unsigned open = __ballot_sync(0xffffffffu, q >= 0);
      const int base = open ? __shfl_sync(0xffffffffu, q - r, __ffs(open) - 1) : 0;
      const int d = q - r - base;
      if (lane == 0) latb[(size_t)w * NL + j] = base;
      if (home)
        latd[(size_t)r * NL + j] =
            (short)(q < 0 ? kLatClosed : (d < -32000 || d > 32000 ? kLatWide : d));
    }
  }
}

// The face coefficients of np_cell: species k's at co[k * (DIM + 1) * n + ...].
template <int DIM>
__global__ void k_np_coef64(const NFlag *__restrict__ fl, const int *__restrict__ lat, int n,
                            const double *__restrict__ u, const double *__restrict__ phi,
                            NPConst<double> c, int ns, double2 *__restrict__ co) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    const unsigned f = fl[r];
    const double phP = phi[r];
    auto put = [&](int a, double uf, double dd) {
      for (int k = 0; k < ns; k++) {
        double Bp, Bm;
        bernoulli_pair(r_fma(-c.zf[k], dd, r_mul(uf, c.dxD[k])), Bp, Bm);
        co[((size_t)k * (DIM + 1) + a) * n + r] =
            make_double2(r_mul(c.Ddx[k], Bp), r_mul(c.Ddx[k], Bm));
      }
    };
#pragma unroll
    for (int a = 0; a < DIM; a++) {
      const double uP = u[(size_t)a * n + r];
      const int q = plus_face(f, lat, n, a, r);
      if (q >= 0) put(a, r_mul(0.5, r_add(uP, u[(size_t)a * n + q])), phi_diff(phi[q], phP));
    }
    if ((f >> (kEdgeBit + 1)) & 1u) put(DIM, r_mul(-0.5, r_add(u[r], u[r])), phi_diff(0.0, phP));
  }
}

// One FP64 step of species k at rank r (of all 32 ranks of its warp) and its
// account.
template <int DIM, bool EARLY>
__device__ __forceinline__ void np_step_body(const double *Cin, double *Cout,
                                             const double *__restrict__ u,
                                             const double *__restrict__ phi,
                                             const double2 *__restrict__ co, const NPGeo &g,
                                             const NPConst<double> &c, double *acc, int r, int k) {
  const size_t n = (size_t)g.n;
  double v[3] = {0.0, 0.0, 0.0};
  bool io = false;
  if (r < g.n)
    io = np_cell<DIM, EARLY>(Cin + k * n, Cout + k * n, co ? co + (size_t)k * (DIM + 1) * n : nullptr, u,
                      phi, g, g.fl[r], r, c, k, v);
  if (EARLY) pdl_wait();  // (a warp without cells has not waited yet)
  np_account(v, io, acc + (size_t)(3 * k) * g.naccs, r >> 5, g.naccs);
}

// Has the inputs of the tiles `ahead` of this block's fetched into L2 (one
// thread, a bulk prefetch per array): the records across the high lateral
// face (z+, or y+ in 2D: in rank order the first of a record's five reads;
// the place is displaced as at this block's own tile, which is close enough
// for a hint), the face data, the link data and the account slots.
template <int DIM, int NS, int TILES, bool PAIR>
__device__ __forceinline__ void np_prefetch(const NPFields &F, int n, int naccs, int w,
                                            int ahead) {
  constexpr int NL = 2 * DIM - 2, CELLS = TILES * kHome;
  const int w0 = w + ahead;
  if ((long long)(w0 + 2 * TILES) * kHome >= n) return;
  // whole 16-byte units; at most 15 bytes to either side of the range, which
  // the test above keeps inside the arrays
  auto pre = [](const void *p, unsigned bytes) {
    const unsigned long long at = (unsigned long long)p & ~15ull;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(at), "r"((bytes + 15u) & ~15u)
                 : "memory");
  };
  const size_t r0 = (size_t)w0 * kHome;
  const long long z0 = (long long)r0 + F.latb[(size_t)w * NL + (DIM == 3 ? 2 : 0)];
  if (z0 >= 0 && z0 + 2 * CELLS < n) {
#pragma unroll
    for (int p = 0; p < (NS + 1) / 2; p++) {
      constexpr unsigned words = PAIR ? 2u : 1u;
      const unsigned rec = (2 * p + 1 < NS ? 8u : 4u) * words;
      pre((const char *)F.C[p] + (size_t)z0 * rec, CELLS * rec);
    }
  }
#pragma unroll
  for (int a = 0; a < DIM; a++) pre(F.fd[a] + r0, CELLS * 8u);
  pre(F.latd + r0 * NL, CELLS * NL * 2u);
  pre(F.fl + r0, CELLS * 2u);
  pre(F.latb + (size_t)w0 * NL, TILES * NL * 4u);
#pragma unroll
  for (int k = 0; k < NS; k++) pre(F.acc + (size_t)(3 * k) * naccs + w0, TILES * 8u);
}

// FP32 storage: warps of 31 home cells (np_warp31); ahead > 0: np_prefetch.
// 256^3 pack, pair concentrations: 231 -> 141 us a step (1.6 -> 2.6 TB/s of the
// method's 49 bytes a cell), 1024x512: 6.7 -> 6.0, before early launches
// (launch_pdl: 138 and 5.1 us).
template <int DIM, int NS, int BS, bool PAIR, int MODE>
__global__ void __launch_bounds__(BS)
    k_np_step32(const __grid_constant__ NPFields F, int n, int naccs,
                const __grid_constant__ NPConst<float> c, int ahead) {
  const int w = (int)((blockIdx.x * BS + threadIdx.x) >> 5);
  if (ahead > 0 && threadIdx.x == 0) np_prefetch<DIM, NS, BS / 32, PAIR>(F, n, naccs, w, ahead);
  np_warp31<DIM, NS, PAIR, MODE, true>(F, n, naccs, c, w);
}

// FP64 storage, one thread per pore cell and species (blockIdx.y).
template <int DIM, int BS>
__global__ void __launch_bounds__(BS)
    k_np_step(const double *Cin, double *Cout,
              const double *__restrict__ u, const double *__restrict__ phi,
              const double2 *__restrict__ co, NPGeo g, NPConst<double> c,
              double *acc) {
  np_step_body<DIM, true>(Cin, Cout, u, phi, co, g, c, acc, (int)(blockIdx.x * BS + threadIdx.x),
                    (int)blockIdx.y);
}

// One member of a fused sweep: its own concentrations, velocity, potential,
// constants (time step) and accounts.
template <typename T> struct SweepMember {
  T *C[2];          // concentration buffers (ping-pong)
  NPFields f[2];    // FP32: the fields of a step from buffer 0 / 1
  const T *u;
  const typename PhiStore<T>::type *phi;
  const double2 *co;  // FP64: face coefficients (null: evaluated at every step)
  typename AccSlot<T>::type *acc;
  NPConst<T> c;
};

// (Sweep and batch steps follow one another in full order, EARLY = false: over
// their many waves the gap between launches is a small share of a step.)
//
// All members of a sweep advance one step in one launch: block (b, m) runs
// the cells of block b for member m (the block -> cells map, the arithmetic
// and the accounts of a member are those of a single run's launch, so a
// member's result equals a single run's bit for bit).
template <typename T, int DIM, int NS, bool PAIR, int MODE>
__global__ void __launch_bounds__(kRowBlock)
    k_np_sweep(const SweepMember<T> *__restrict__ members, int in, NPGeo g) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const SweepMember<T> &mb = members[blockIdx.y];
  if constexpr (std::is_same<T, float>::value)
    np_warp31<DIM, NS, PAIR, MODE, false>(mb.f[in], g.n, g.naccs, mb.c, r >> 5);
  else
    for (int k = 0; k < NS; k++)
      np_step_body<DIM, false>(mb.C[in], mb.C[1 - in], mb.u, mb.phi, mb.co, g, mb.c, mb.acc, r, k);
}

// One member of a batch over several geometries: a sweep member plus its
// geometry; blocks [block0, block0 + nblocks) of the launch are its own.
template <typename T> struct BatchMember {
  SweepMember<T> s;
  NPGeo g;
  int block0, nblocks;
};

// All members of a batch over uneven geometries advance one step in one
// launch.  Block b of the launch belongs to the member whose block range
// holds it (binary search over the ascending block0), and runs that member's
// local block b - block0: the same cells, arithmetic and accounts as block
// b - block0 of the member's single-run launch, so each member equals its
// single run bit for bit.
template <typename T, int DIM, int NS, bool PAIR, int MODE>
__global__ void __launch_bounds__(kRowBlock)
    k_np_batch(const BatchMember<T> *__restrict__ members, int n_members, int in) {
  int lo = 0, hi = n_members - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (members[mid].block0 <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const BatchMember<T> &mb = members[lo];
  const int b = (int)blockIdx.x - mb.block0;
  const int r = b * blockDim.x + threadIdx.x;
  if constexpr (std::is_same<T, float>::value)
    np_warp31<DIM, NS, PAIR, MODE, false>(mb.s.f[in], mb.g.n, mb.g.naccs, mb.s.c, r >> 5);
  else
    for (int k = 0; k < NS; k++)
      np_step_body<DIM, false>(mb.s.C[in], mb.s.C[1 - in], mb.s.u, mb.s.phi, mb.s.co, mb.g, mb.s.c,
                        mb.s.acc, r, k);
}

// Largest outflow rate over pore cells and species, in FP64 from the FP64
// lattice velocity and potential:  (1/dx) [sum_{open faces} (D/dx) B(-P_f)
// + n_solid K_eff]; dt = safety / max.
template <int DIM>
__global__ void __launch_bounds__(kRedThreads)
    k_np_rate(const NFlag *__restrict__ fl, const double *__restrict__ uflow,
              const double *__restrict__ psi, NPConst<double> c, int ns, double scale,
              double inv_vt, double inv_dx, double safety, int nx, int NX, int ny, int nz,
              long long N, long long Nf, int walls, double *__restrict__ part,
              unsigned int *counter, double *scal) {
  __shared__ double sm[32];
  double v[1] = {0.0};
  for (long long P = blockIdx.x * (long long)blockDim.x + threadIdx.x; P < N;
       P += (long long)gridDim.x * blockDim.x) {
    const unsigned f = fl[P];
    if (f & 1u) continue;
    const long long row = P / nx;
    const int x = (int)(P - row * nx);
    const long long sP = row * NX + x;
    for (int k = 0; k < ns; k++) {
      double rate = 0.0;
      for (int fc = 0; fc < 2 * DIM; fc++) {
        const int a = fc >> 1;
        const double sg = (fc & 1) ? -1.0 : 1.0;
        long long Q = 0;
        const int kind = np_face<DIM>(f, fc, nx, ny, nz, walls, P, Q);
        if (kind == F_WALL) continue;
        if (kind == F_SOLID) {
          rate += c.Keff[k];
          continue;
        }
        const double uP = scale * uflow[(size_t)a * Nf + sP];
        double unb = uP, psinb = 0.0;
        const double psiP = psi[P];
        if (kind == F_PORE) {
          const long long rq = Q / nx;
          unb = scale * uflow[(size_t)a * Nf + rq * NX + (Q - rq * nx)];
          psinb = psi[Q];
        } else if (kind == F_OUTLET) {
          psinb = psiP;
        }
        const double Pf = 0.5 * (uP + unb) * sg * c.dxD[k] - c.zf[k] * (psinb - psiP) * inv_vt;
        double Bp, Bm;
        bernoulli_pair(Pf, Bp, Bm);
        rate += c.Ddx[k] * Bm;
      }
      v[0] = fmax(v[0], rate * inv_dx);
    }
  }
  block_reduce<1>(v, sm, OpMax(), 0.0);
  if (threadIdx.x == 0) part[blockIdx.x] = v[0];
  if (last_block(counter, gridDim.x)) {
    combine_partials<1>(part, gridDim.x, v, sm, OpMax(), 0.0);
    if (threadIdx.x == 0) {
      scal[S_RATE] = v[0];
      scal[S_DT] = v[0] > 0.0 ? safety / v[0] : 0.0;
      *counter = 0;
    }
  }
}

// The saturated start: every cell of species k at c0 (hi + lo).
template <typename T>
__global__ void k_np_init(CViews<T> C, int n, int ns, T c0, T c0lo) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x)
    for (int k = 0; k < ns; k++) {
      T *p = const_cast<T *>(C.v[k].p) + (size_t)r * C.v[k].stride;
      p[0] = c0;
      if (C.v[k].lo) p[C.v[k].lo] = c0lo;
    }
}

// Dissolved amount, outlet sums (flux weighted and plain) per species.
// Values: [0,4) mass, [4,8) sum u_x C at the outlet, 8 sum u_x, [9,13) plain
// sum of C at the outlet, 13 pore cells in the outlet column.
template <typename T>
__global__ void __launch_bounds__(kRedThreads)
    k_np_sums(const NFlag *__restrict__ fl, CViews<T> C, const T *__restrict__ u, int n,
              int ns, double cell_vol, double *__restrict__ part, unsigned int *counter, double *scal) {
  constexpr int NV = 14;
  __shared__ double sm[NV * 32];
  double v[NV];
#pragma unroll
  for (int j = 0; j < NV; j++) v[j] = 0.0;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    const bool outlet = ((unsigned)fl[r] >> kEdgeBit) & 1u;
    const double ux = (double)u[r];
#pragma unroll
    for (int k = 0; k < kMaxSpecies; k++) {
      if (k >= ns) break;
      const double ck = C.v[k].at(r);
      v[k] += ck;
      if (outlet) {
        v[4 + k] += ux * ck;
        v[9 + k] += ck;
      }
    }
    if (outlet) {
      v[8] += ux;
      v[13] += 1.0;
    }
  }
  block_reduce<NV>(v, sm, OpSum(), 0.0);
  if (threadIdx.x == 0)
#pragma unroll
    for (int j = 0; j < NV; j++) part[(size_t)j * gridDim.x + blockIdx.x] = v[j];
  if (last_block(counter, gridDim.x)) {
    combine_partials<NV>(part, gridDim.x, v, sm, OpSum(), 0.0);
    if (threadIdx.x == 0) {
      for (int k = 0; k < kMaxSpecies; k++) {
        scal[S_MASS + k] = v[k] * cell_vol;
        scal[S_OUT + 2 * k] = v[4 + k];
        scal[S_OUT + 2 * k + 1] = v[8];
        scal[S_OUTP + k] = v[9 + k];
      }
      scal[S_OUTN] = v[13];
      *counter = 0;
    }
  }
}

// Pore cells and pore-solid faces inside the image (the interface the
// specific surface of Sec. 4 measures), counted over the pore ranks, and the
// sum of the x velocity over them (the numerator of Sec. 4's pore mean U).
template <typename T>
__global__ void __launch_bounds__(kRedThreads)
    k_geometry(const NFlag *__restrict__ fl, const T *__restrict__ ux, int n, int faces,
               double *__restrict__ part, unsigned int *counter, double *scal) {
  __shared__ double sm[3 * 32];
  double v[3] = {0.0, 0.0, 0.0};
  const unsigned face_bits = ((1u << faces) - 1u) << kFaceBit;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    v[0] += 1.0;
    v[1] += (double)__popc((unsigned)fl[r] & face_bits);
    v[2] += (double)ux[r];
  }
  block_reduce<3>(v, sm, OpSum(), 0.0);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = v[0];
    part[gridDim.x + blockIdx.x] = v[1];
    part[2 * gridDim.x + blockIdx.x] = v[2];
  }
  if (last_block(counter, gridDim.x)) {
    combine_partials<3>(part, gridDim.x, v, sm, OpSum(), 0.0);
    if (threadIdx.x == 0) {
      scal[S_GEOM] = v[0];
      scal[S_GEOM + 1] = v[1];
      scal[S_GEOM + 2] = v[2];
      *counter = 0;
    }
  }
}

// Totals of the per-warp Gamma/In/Out accounts (one block, fixed order).
template <typename A>
__global__ void __launch_bounds__(kRedThreads)
    k_acc_total(const A *__restrict__ acc, int nw, double *scal) {
  constexpr int NV = 3 * kMaxSpecies;
  __shared__ double sm[NV * 32];
  double v[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) v[k] = 0.0;
  for (int b = threadIdx.x; b < nw; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] += acc_value(acc[(size_t)k * nw + b]);
  block_reduce<NV>(v, sm, OpSum(), 0.0);
  if (threadIdx.x == 0)
#pragma unroll
    for (int j = 0; j < NV; j++) scal[S_ACC + j] = v[j];
}

// Launches k_acc_total for the domain's precision.
void acc_total(const cdi_domain *d, const void *acc, cudaStream_t st, double *scal) {
  if (d->prec == CDI_FP64)
    k_acc_total<double><<<1, kRedThreads, 0, st>>>((const double *)acc, d->np_accs, scal);
  else
    k_acc_total<float2><<<1, kRedThreads, 0, st>>>((const float2 *)acc, d->np_accs, scal);
}

// Mean of species k over the pore cells of each x column (the column's
// cells found through the row words).
template <typename T>
__global__ void __launch_bounds__(kRedThreads)
    k_colmeans(const uint2 *__restrict__ words, int W, CView<T> C, int rows,
               double *__restrict__ out) {
  __shared__ double sm[2 * 32];
  const int x = blockIdx.x;
  double v[2] = {0.0, 0.0};
  for (int row = threadIdx.x; row < rows; row += blockDim.x) {
    const uint2 t = words[(size_t)row * W + (x >> 5)];
    if (!((t.y >> (x & 31)) & 1u)) continue;
    const int r = t.x + __popc(t.y & ((1u << (x & 31)) - 1u));
    v[0] += C.at(r);
    v[1] += 1.0;
  }
  block_reduce<2>(v, sm, OpSum(), 0.0);
  if (threadIdx.x == 0) out[x] = v[1] > 0.0 ? v[0] / v[1] : 0.0;
}

// Per pore rank and lateral face (y+, y-, z+, z-): the rank of the pore
// neighbour across it (rows wrap periodically), or -1 across a solid face or
// a lateral wall.  The step kernels read it instead of the row words, which
// saves them a dependent load and the rank arithmetic.
__global__ void k_lat_nbr(const NFlag *__restrict__ fl, const int *__restrict__ cells,
                          const uint2 *__restrict__ words, int n, int nx, int W, int ny, int nz,
                          int walls, int faces, int *__restrict__ lat) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    const unsigned f = fl[r];
    const int P = cells[r], row = P / nx, x = P - row * nx;
    for (int fc = 2; fc < faces; fc++) {
      const bool solid = (f >> (kFaceBit + fc)) & 1u;
      const bool wall = ((f >> (kEdgeBit + fc)) & 1u) && walls;
      lat[(size_t)(fc - 2) * n + r] =
          (solid || wall) ? -1 : rank_of(words, W, lateral_row(f, fc, row, ny, nz), x);
    }
  }
}

// Per pore rank: its face flags.
__global__ void k_cfl(const NFlag *__restrict__ fl, const int *__restrict__ cells, int n,
                      NFlag *__restrict__ cfl) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x)
    cfl[r] = fl[cells[r]];
}

// Per 32 cells of a row: the pore bits and the rank of the first pore cell at
// or after the word's first cell (binary search of the ascending cell list).
__global__ void k_words(const NFlag *__restrict__ fl, const int *__restrict__ cells, int n,
                        int nx, int W, long long n_words, uint2 *__restrict__ words) {
  for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < n_words;
       w += (long long)gridDim.x * blockDim.x) {
    const long long row = w / W;
    const int x0 = (int)(w - row * W) * 32;
    const long long P0 = row * nx + x0;
    unsigned bits = 0;
    for (int b = 0; b < 32 && x0 + b < nx; b++)
      if (!(fl[P0 + b] & 1u)) bits |= 1u << b;
    int lo = 0, hi = n;  // first rank with cells[rank] >= P0
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((long long)cells[mid] < P0) lo = mid + 1;
      else hi = mid;
    }
    words[w] = make_uint2((unsigned)lo, bits);
  }
}

// Compact (rank-ordered) fields -> FP64 lattice fields, 0 in solid cells:
// dst[a * N + cells[r]] = the value of component a at rank r.
template <typename T>
__global__ void k_scatter(CViews<T> src, int comps, const int *__restrict__ cells, int n,
                          long long N, double *__restrict__ dst) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    const long long P = cells[r];
    for (int a = 0; a < comps; a++) dst[a * N + P] = src.v[a].at(r);
  }
}

// Species records <-> planes of kMaxSpecies hi words followed (pair storage)
// by kMaxSpecies lo words, the order of a saved state; the planes of absent
// species are 0.
__global__ void k_records_to_planes(CViews<float> C, int n, int ns, float *__restrict__ hi,
                                    float *__restrict__ lo) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x)
    for (int k = 0; k < kMaxSpecies; k++) {
      const float *p = k < ns ? C.v[k].p + (size_t)r * C.v[k].stride : nullptr;
      hi[(size_t)k * n + r] = p ? p[0] : 0.f;
      if (lo) lo[(size_t)k * n + r] = p ? p[C.v[k].lo] : 0.f;
    }
}
__global__ void k_planes_to_records(CViews<float> C, int n, int ns, const float *__restrict__ hi,
                                    const float *__restrict__ lo) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x)
    for (int k = 0; k < ns; k++) {
      float *p = const_cast<float *>(C.v[k].p) + (size_t)r * C.v[k].stride;
      p[0] = hi[(size_t)k * n + r];
      if (lo) p[C.v[k].lo] = lo[(size_t)k * n + r];
    }
}

template <typename T> NPConst<T> make_const(const cdi_domain *d) {
  NPConst<T> c{};
  for (int k = 0; k < kMaxSpecies; k++) {
    c.dxD[k] = (T)(d->dx / d->D[k]);
    c.Ddx[k] = (T)(d->D[k] / d->dx);
    c.Keff[k] = (T)(d->Ka / (1.0 + d->Ka * d->dx / (2.0 * d->D[k])));
    c.zf[k] = (T)d->z[k];
  }
  c.dtdx = (T)(d->dt / d->dx);
  c.c0 = (T)d->c0;
  c.c0lo = (T)(d->c0 - (double)c.c0);
  return c;
}

// The FP32 fields of a transport state (stepping from Cin into Cout; fd the
// face data of its velocity and potential).
NPFields fields32(const cdi_domain *d, const void *Cin, void *Cout, const float2 *fd,
                  const float2 *bern, const void *u, const void *phi, void *acc) {
  NPFields F{};
  const size_t n = (size_t)d->n_pore, pair = 2 * n * (d->cpair ? 2 : 1);
  for (int p = 0; p < 2; p++) {
    F.C[p] = (const float *)Cin + p * pair;
    F.Co[p] = (float *)Cout + p * pair;
  }
  for (int a = 0; a < d->dim; a++) F.fd[a] = fd + (size_t)a * n;
  F.latd = d->d_latd;
  F.latb = d->d_latb;
  F.lat = d->d_latnb;
  F.ux = (const float *)u;
  F.phi = (const float2 *)phi;
  F.fl = d->d_cfl;
  F.bern = bern;
  F.acc = (float2 *)acc;
  return F;
}

// The face data of velocity u and potential phi (FP32 storage); *any_large
// (device, cleared by the caller) tells whether a face has |P| >= 1/2.
void launch_faces(const cdi_domain *d, cudaStream_t st, const void *u, const void *phi,
                  float2 *fd, int *any_large) {
  const int n = (int)d->n_pore, grid = std::min((n + 255) / 256, 16 * kRedBlocks);
  const NPConst<float> c = make_const<float>(d);
  auto *kern = d->dim == 2 ? k_np_faces<2> : k_np_faces<3>;
  kern<<<grid, 256, 0, st>>>(d->d_cfl, d->d_latnb, n, (const float *)u, (const float2 *)phi, c,
                             d->ns, fd, any_large);
}
void launch_bern(const cdi_domain *d, cudaStream_t st, const void *u, const void *phi,
                 const float2 *fd, float2 *bern) {
  const int n = (int)d->n_pore, grid = std::min((n + 255) / 256, 16 * kRedBlocks);
  const NPConst<float> c = make_const<float>(d);
  auto *kern = d->dim == 2 ? k_np_bern<2> : k_np_bern<3>;
  kern<<<grid, 256, 0, st>>>(d->d_cfl, d->d_latnb, n, (const float *)u, (const float2 *)phi, fd, c,
                             d->ns, bern);
}
void launch_coef64(const cdi_domain *d, cudaStream_t st, const void *u, const void *phi,
                   void *co) {
  const int n = (int)d->n_pore, grid = std::min((n + 127) / 128, 16 * kRedBlocks);
  auto *kern = d->dim == 2 ? k_np_coef64<2> : k_np_coef64<3>;
  kern<<<grid, 128, 0, st>>>(d->d_cfl, d->d_latnb, n, (const double *)u, (const double *)phi,
                             make_const<double>(d), d->ns, (double2 *)co);
}
// Bytes of the stored Bernoulli pairs (FP32) or face coefficients (FP64).
size_t bern_bytes(const cdi_domain *d) {
  return (size_t)(d->dim + 1) * d->n_pore * d->ns *
         (d->prec == CDI_FP64 ? sizeof(double2) : sizeof(float2));
}

NPGeo make_geo(const cdi_domain *d) {
  return NPGeo{d->d_cfl, d->d_latnb, (int)d->n_pore, d->np_accs};
}

// Tiles between a block and the ones whose inputs it has fetched into L2: one
// to two waves of resident warps.  0 (no prefetch) where a step's whole
// working set stays in L2 from one step to the next.
int np_ahead_tiles(const cdi_domain *d) {
  const size_t rec = (size_t)d->ns * (d->cpair ? 8 : 4);
  const size_t step = (size_t)d->n_pore * (2 * rec + d->dim * 8 + 4 * (d->dim - 1) + 2);
  return step > ((size_t)96 << 20) ? 8192 : 0;
}

// dep: the launch before this one in the stream is a step too, so this one may
// start early (launch_pdl).  Behind anything else a step starts in full order:
// it reads face data and member tables ahead of its wait.
template <typename T, int DIM, int NS, int BS, bool PAIR>
void launch_step_bs(cdi_domain *d, cudaStream_t st, int in, bool dep) {
  // FP64: one thread per pore rank; FP32: warps of 31 home cells (one
  // account set per warp either way)
  const long long units = std::is_same<T, float>::value ? np_warps(d->n_pore) * 32 : d->n_pore;
  const int grid = (int)((units + BS - 1) / BS);
  if constexpr (std::is_same<T, float>::value) {
    const NPFields F = fields32(d, d->d_C[in], d->d_C[1 - in], d->d_fd, (const float2 *)d->d_bern, d->d_u,
                                d->d_phi, d->d_acc);
    auto *kern = d->np_mode == NP_SMALL   ? k_np_step32<DIM, NS, BS, PAIR, NP_SMALL>
                 : d->np_mode == NP_LARGE ? k_np_step32<DIM, NS, BS, PAIR, NP_LARGE>
                                          : k_np_step32<DIM, NS, BS, PAIR, NP_EVAL>;
    launch_pdl(kern, grid, BS, st, dep, F, (int)d->n_pore, d->np_accs, make_const<float>(d),
               np_ahead_tiles(d));
  } else {
    launch_pdl(k_np_step<DIM, BS>, dim3(grid, NS), BS, st, dep, (const double *)d->d_C[in],
               (double *)d->d_C[1 - in], (const double *)d->d_u, (const double *)d->d_phi,
               d->np_mode == NP_EVAL ? nullptr : (const double2 *)d->d_bern, make_geo(d),
               make_const<double>(d), d->d_acc);
  }
}

template <typename T, int DIM, int NS, bool PAIR>
void launch_step_t(cdi_domain *d, cudaStream_t st, int in, bool dep) {
  switch (d->np_block) {
    case 64: launch_step_bs<T, DIM, NS, 64, PAIR>(d, st, in, dep); break;
    case 256: launch_step_bs<T, DIM, NS, 256, PAIR>(d, st, in, dep); break;
    default: launch_step_bs<T, DIM, NS, 128, PAIR>(d, st, in, dep); break;
  }
}

template <typename T, int DIM, bool PAIR>
void launch_step_d(cdi_domain *d, cudaStream_t st, int in, bool dep) {
  switch (d->ns) {
    case 1: launch_step_t<T, DIM, 1, PAIR>(d, st, in, dep); break;
    case 2: launch_step_t<T, DIM, 2, PAIR>(d, st, in, dep); break;
    case 3: launch_step_t<T, DIM, 3, PAIR>(d, st, in, dep); break;
    default: launch_step_t<T, DIM, 4, PAIR>(d, st, in, dep); break;
  }
}

void launch_step(cdi_domain *d, cudaStream_t st, int in, bool dep) {
  if (d->prec == CDI_FP64) {
    if (d->dim == 2) launch_step_d<double, 2, false>(d, st, in, dep);
    else launch_step_d<double, 3, false>(d, st, in, dep);
  } else if (d->cpair) {
    if (d->dim == 2) launch_step_d<float, 2, true>(d, st, in, dep);
    else launch_step_d<float, 3, true>(d, st, in, dep);
  } else {
    if (d->dim == 2) launch_step_d<float, 2, false>(d, st, in, dep);
    else launch_step_d<float, 3, false>(d, st, in, dep);
  }
}

constexpr int kGraphSteps = 64;  // steps per captured transport graph (even)

// Launch shapes: 64, 128 or 256 threads per block (0-2); 3-9 name the default
// again.  128 is taken unless a shape is fixed: it is the fastest or within
// 4 % of it on every size measured (before early launches, us a step for 64 /
// 128 / 256: 256^3 155 / 139 / 154; 1024x512 5.8 / 5.8 / 5.9; 96^3 11.3 / 10.6 /
// 11.1; FP64 128x64 4.0 / 4.0 / 4.9), so no launch is spent on timing
// candidates.  Accounts are kept per warp whatever the shape, so every choice
// computes the same bits.
constexpr int kNpDefaultShape = 1;
constexpr int kNpVariantBlock[10] = {64, 128, 256, 128, 128, 128, 128, 128, 128, 128};

}  // namespace

int cdi_np_shape_block(int v) { return v >= 0 && v < 10 ? kNpVariantBlock[v] : 0; }

cdi_status cdi_np_build_flags(cdi_domain *d) {
  dim3 grid((d->nx + kRowBlock - 1) / kRowBlock, d->ny, d->nz);
  if (d->dim == 2)
    k_np_flags<2><<<grid, kRowBlock, 0, d->stream>>>(d->d_mask, d->d_nflags, d->nx, d->ny, d->nz,
                                                     d->walls);
  else
    k_np_flags<3><<<grid, kRowBlock, 0, d->stream>>>(d->d_mask, d->d_nflags, d->nx, d->ny, d->nz,
                                                     d->walls);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "face flags");
  return CDI_OK;
}

cdi_status cdi_np_init(cdi_domain *d, double dt_s, double *dt_used) {
  if (d->np_graph) cudaGraphExecDestroy(d->np_graph);
  d->np_graph = nullptr;
  d->imp_stale = d->faces_stale = true;  // they follow u, phi and the species
  double dt = dt_s;
  if (dt <= 0.0) {
    cdi_status s = cdi_np_dt(d, d->h_scal[S_SCALE], &dt);
    if (s != CDI_OK) return s;
  }
  d->dt = dt;
  if (dt_used) *dt_used = dt;
  if (!(d->imp_tol > 0.0)) {  // (implicit steps do not read them)
    cdi_status fs = cdi_np_faces(d);
    if (fs != CDI_OK) return fs;
  }
  if (!d->np_tuned) {
    d->np_variant = kNpDefaultShape;
    d->np_block = kNpVariantBlock[d->np_variant];
    d->np_tuned = true;
  }
  if (d->prec == CDI_FP64)
    k_np_init<double><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        c_views<double>(d, d->d_C[0]), (int)d->n_pore, d->ns, d->c0, 0.0);
  else
    k_np_init<float><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        c_views<float>(d, d->d_C[0]), (int)d->n_pore, d->ns, (float)d->c0,
        (float)(d->c0 - (double)(float)d->c0));
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "transport init");
  CDI_TRY(d, cudaMemsetAsync(d->d_acc, 0, (size_t)3 * kMaxSpecies * d->np_accs * 8, d->stream),
          "reset accumulators");
  d->cur = 0;
  d->np_steps = 0;
  return CDI_OK;
}

// Memory for the domain's Bernoulli pairs or face coefficients (kept for its
// life); false when there is none.
static bool take_bern(cdi_domain *d) {
  if (d->d_bern && d->bern_bytes < bern_bytes(d)) {
    cudaStreamSynchronize(d->stream);  // steps in flight read it
    cdi_dev_release(d, d->d_bern);
    d->d_bern = nullptr;
  }
  if (!d->d_bern) {
    d->bern_bytes = bern_bytes(d);
    d->d_bern = cdi_dev_alloc(d, d->bern_bytes);
  }
  return d->d_bern != nullptr;
}

// What the step keeps of the domain's current velocity and potential (after
// either, or the species, has changed).  FP64: the face coefficients.  FP32:
// the face data, and the Bernoulli pairs where some face needs them (their
// memory is taken the first time one does; waits for the stream).  Without
// memory for them the step evaluates every face itself.
static cdi_status form_faces(cdi_domain *d) {
  if (d->prec == CDI_FP64) {
    d->np_mode = take_bern(d) ? NP_SMALL : NP_EVAL;
    if (d->np_mode == NP_EVAL) return CDI_OK;
    launch_coef64(d, d->stream, d->d_u, d->d_phi, d->d_bern);
    d->timing.kernel_launches++;
    CDI_TRY(d, cudaGetLastError(), "face coefficients");
    return CDI_OK;
  }
  int *flag = (int *)(d->d_counter + C_FACE);
  int large = 0;
  CDI_TRY(d, cudaMemsetAsync(flag, 0, sizeof(int), d->stream), "face flag reset");
  launch_faces(d, d->stream, d->d_u, d->d_phi, d->d_fd, flag);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "face data");
  CDI_TRY(d, cudaMemcpyAsync(&large, flag, sizeof(int), cudaMemcpyDeviceToHost, d->stream),
          "face flag");
  CDI_TRY(d, cudaStreamSynchronize(d->stream), "face data");
  d->np_mode = large ? (take_bern(d) ? NP_LARGE : NP_EVAL) : NP_SMALL;
  if (d->np_mode != NP_LARGE) return CDI_OK;
  launch_bern(d, d->stream, d->d_u, d->d_phi, d->d_fd, (float2 *)d->d_bern);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "face data");
  return CDI_OK;
}
cdi_status cdi_np_faces(cdi_domain *d) {
  // captured steps hold the mode and the memory of the faces before
  if (d->np_graph) cudaGraphExecDestroy(d->np_graph);
  d->np_graph = nullptr;
  const cdi_status s = form_faces(d);
  d->faces_stale = s != CDI_OK;
  return s;
}

// Explicit time step for the current potential (d_psi) and the solved flow
// scaled by `scale` (the species set in the domain).
cdi_status cdi_np_dt(cdi_domain *d, double scale, double *dt_out) {
  double dt = 0.0;
  {
    NPConst<double> c = make_const<double>(d);
    if (d->dim == 2)
      k_np_rate<2><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
          d->d_nflags, d->d_uflow, d->d_psi, c, d->ns, scale, 1.0 / d->VT, 1.0 / d->dx, 0.9,
          d->nx, d->NX, d->ny, d->nz, d->N, d->Nf, d->walls, d->d_part, d->d_counter + C_DT,
          d->d_scal);
    else
      k_np_rate<3><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
          d->d_nflags, d->d_uflow, d->d_psi, c, d->ns, scale, 1.0 / d->VT, 1.0 / d->dx, 0.9,
          d->nx, d->NX, d->ny, d->nz, d->N, d->Nf, d->walls, d->d_part, d->d_counter + C_DT,
          d->d_scal);
    d->timing.kernel_launches++;
    CDI_TRY(d, cudaGetLastError(), "time step kernel");
    CDI_TRY(d, cudaMemcpyAsync(d->h_scal + S_RATE, d->d_scal + S_RATE, 2 * sizeof(double),
                               cudaMemcpyDeviceToHost, d->stream),
            "time step copy");
    CDI_TRY(d, cudaStreamSynchronize(d->stream), "time step");
    dt = d->h_scal[S_DT];
    if (!(dt > 0.0) || !std::isfinite(dt))
      return cdi_fail(d, CDI_ERR_INVALID_ARG, "no finite time step (no flux anywhere?)");
  }
  *dt_out = dt;
  return CDI_OK;
}

// ---------------------------------------------------------------------------
// Fused sweep: n members on one geometry, one launch per step for all.
// ---------------------------------------------------------------------------
namespace {

template <typename T, int DIM, bool PAIR, int MODE>
void launch_sweep_d(cdi_domain *d, cudaStream_t st, const void *members, int n, int in) {
  const SweepMember<T> *m = (const SweepMember<T> *)members;
  const NPGeo g = make_geo(d);
  const dim3 grid(d->np_blocks, n);
  switch (d->ns) {
    case 1: k_np_sweep<T, DIM, 1, PAIR, MODE><<<grid, kRowBlock, 0, st>>>(m, in, g); break;
    case 2: k_np_sweep<T, DIM, 2, PAIR, MODE><<<grid, kRowBlock, 0, st>>>(m, in, g); break;
    case 3: k_np_sweep<T, DIM, 3, PAIR, MODE><<<grid, kRowBlock, 0, st>>>(m, in, g); break;
    default: k_np_sweep<T, DIM, 4, PAIR, MODE><<<grid, kRowBlock, 0, st>>>(m, in, g); break;
  }
}

template <int DIM, bool PAIR>
void launch_sweep32(cdi_domain *d, cudaStream_t st, const void *members, int n, int in,
                    int mode) {
  if (mode == NP_SMALL) launch_sweep_d<float, DIM, PAIR, NP_SMALL>(d, st, members, n, in);
  else if (mode == NP_LARGE) launch_sweep_d<float, DIM, PAIR, NP_LARGE>(d, st, members, n, in);
  else launch_sweep_d<float, DIM, PAIR, NP_EVAL>(d, st, members, n, in);
}

void launch_sweep(cdi_domain *d, cudaStream_t st, const void *members, int n, int in, int mode) {
  if (d->prec == CDI_FP64) {
    if (d->dim == 2) launch_sweep_d<double, 2, false, NP_SMALL>(d, st, members, n, in);
    else launch_sweep_d<double, 3, false, NP_SMALL>(d, st, members, n, in);
  } else if (d->cpair) {
    if (d->dim == 2) launch_sweep32<2, true>(d, st, members, n, in, mode);
    else launch_sweep32<3, true>(d, st, members, n, in, mode);
  } else {
    if (d->dim == 2) launch_sweep32<2, false>(d, st, members, n, in, mode);
    else launch_sweep32<3, false>(d, st, members, n, in, mode);
  }
}

// Face data of a member (its own arrays, named in its two field sets), and
// its Bernoulli pairs where a face needs them (false: no memory for them).
void member_faces(const cdi_domain *d, cudaStream_t st, NPFields (&f)[2], const void *u,
                  int *count) {
  launch_faces(d, st, u, f[0].phi, const_cast<float2 *>(f[0].fd[0]), count);
}
bool member_bern(const cdi_domain *d, cudaStream_t st, NPFields (&f)[2], const void *u,
                 void *bern) {
  if (!bern) return false;
  launch_bern(d, st, u, f[0].phi, f[0].fd[0], (float2 *)bern);
  f[0].bern = f[1].bern = (const float2 *)bern;
  return true;
}

template <typename T>
cdi_status sweep_run(cdi_domain *d, int n, const double *scale, const int *group,
                     void *const *phi_groups, const double *dts, int64_t n_steps,
                     double *gamma, double *cout) {
  const size_t TN = (size_t)d->n_pore * sizeof(T);
  const int ns = d->ns;
  const bool f64 = d->prec == CDI_FP64;
  // per-member device memory: velocity, two concentration buffers, accounts
  std::vector<void *> blocks;
  auto take = [&](size_t bytes, bool need = true) {
    void *p = need ? cdi_dev_need(d, bytes) : cdi_dev_alloc(d, bytes);
    if (p) blocks.push_back(p);
    return p;
  };
  std::vector<SweepMember<T>> hm(n);
  bool ok = true;
  for (int m = 0; m < n && ok; m++) {
    void *u = take((size_t)d->dim * TN);
    const size_t CN = (size_t)ns * TN * (d->cpair ? 2 : 1);
    void *c0 = take(CN), *c1 = take(CN);
    void *acc = take((size_t)3 * kMaxSpecies * d->np_accs * 8);
    float2 *fd = f64 ? nullptr : (float2 *)take((size_t)d->dim * d->n_pore * sizeof(float2));
    if (!fd && m == 0) fd = d->d_fd;  // the domain's own state is replaced
    ok = u && c0 && c1 && acc && (f64 || fd);
    if (!ok) break;
    d->dt = dts[m];
    hm[m].C[0] = (T *)c0;
    hm[m].C[1] = (T *)c1;
    for (int in = 0; in < 2; in++)
      hm[m].f[in] = fields32(d, in ? c1 : c0, in ? c0 : c1, fd, nullptr, u,
                             phi_groups[group[m]], acc);
    hm[m].u = (const T *)u;
    hm[m].phi = (const typename PhiStore<T>::type *)phi_groups[group[m]];
    hm[m].acc = (typename AccSlot<T>::type *)acc;
    hm[m].c = make_const<T>(d);
  }
  void *dmem = ok ? take(sizeof(SweepMember<T>) * n) : nullptr;
  int *count = dmem ? (int *)take(sizeof(int) * n) : nullptr;  // a face with |P| >= 1/2, per member
  if (!count) dmem = nullptr;
  cdi_status s = CDI_OK;
  if (!ok || !dmem) s = cdi_fail(d, CDI_ERR_OOM, "sweep: device allocation failed");
  if (s == CDI_OK && cudaMemsetAsync(count, 0, sizeof(int) * n, d->stream) != cudaSuccess)
    s = cdi_fail(d, CDI_ERR_CUDA, "sweep: memset");
  for (int m = 0; m < n && s == CDI_OK; m++) {
    s = cdi_flow_scale_to(d, scale[m], (void *)hm[m].u);
    if (s != CDI_OK) break;
    if (f64) {
      void *co = take(bern_bytes(d), false);
      if (co) launch_coef64(d, d->stream, hm[m].u, hm[m].phi, co);
      hm[m].co = (const double2 *)co;
    } else {
      member_faces(d, d->stream, hm[m].f, hm[m].u, count + m);
    }
    k_np_init<T><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        c_views<T>(d, hm[m].C[0]), (int)d->n_pore, ns, (T)d->c0, (T)(d->c0 - (double)(T)d->c0));
    d->timing.kernel_launches += 2;
    if (cudaMemsetAsync(hm[m].acc, 0, (size_t)3 * kMaxSpecies * d->np_accs * 8, d->stream) !=
        cudaSuccess)
      s = cdi_fail(d, CDI_ERR_CUDA, "sweep: memset");
  }
  int mode = NP_SMALL;
  if (s == CDI_OK && !f64) {
    std::vector<int> large(n);
    if (cudaMemcpyAsync(large.data(), count, sizeof(int) * n, cudaMemcpyDeviceToHost,
                        d->stream) != cudaSuccess || cudaStreamSynchronize(d->stream) != cudaSuccess)
      s = cdi_fail(d, CDI_ERR_CUDA, "sweep: face data");
    for (int m = 0; m < n && s == CDI_OK; m++)
      if (large[m])
        mode = member_bern(d, d->stream, hm[m].f, hm[m].u, take(bern_bytes(d), false))
                   ? std::max<int>(mode, NP_LARGE) : NP_EVAL;
  }
  if (s == CDI_OK &&
      cudaMemcpyAsync(dmem, hm.data(), sizeof(SweepMember<T>) * n, cudaMemcpyHostToDevice,
                      d->stream) != cudaSuccess)
    s = cdi_fail(d, CDI_ERR_CUDA, "sweep: member table");
  // steps: graphs of kGraphSteps fused launches (even, so the parity returns)
  cudaGraphExec_t exec = nullptr;
  int64_t done = 0;
  if (s == CDI_OK) {
    cudaEvent_t ev;
    cdi_timing_begin(d, &ev);
    if (n_steps >= kGraphSteps) {
      cudaGraph_t graph;
      cudaError_t e = cudaStreamBeginCapture(d->cap_stream, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        for (int k = 0; k < kGraphSteps; k++) launch_sweep(d, d->cap_stream, dmem, n, k & 1, mode);
        e = cudaStreamEndCapture(d->cap_stream, &graph);
      }
      if (e == cudaSuccess) {
        e = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
      }
      if (e != cudaSuccess) s = cdi_cuda_fail(d, e, "sweep graph");
      while (s == CDI_OK && n_steps - done >= kGraphSteps) {
        e = cudaGraphLaunch(exec, d->stream);
        if (e != cudaSuccess) s = cdi_cuda_fail(d, e, "sweep graph launch");
        done += kGraphSteps;
      }
    }
    for (; s == CDI_OK && done < n_steps; done++) launch_sweep(d, d->stream, dmem, n, (int)(done & 1), mode);
    cudaError_t e = cudaGetLastError();
    if (s == CDI_OK && e != cudaSuccess) s = cdi_cuda_fail(d, e, "sweep step");
    cdi_timing_end(d, ev, PH_NP, n_steps);
    d->timing.kernel_launches += n_steps;
  }
  // outputs per member, through the same reductions as a single run
  const int cur = (int)(n_steps & 1);
  const double area = d->dim == 2 ? d->dx : d->dx * d->dx;
  const double vol = d->dim == 2 ? d->dx * d->dx : d->dx * d->dx * d->dx;
  for (int m = 0; m < n && s == CDI_OK; m++) {
    k_np_sums<T><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        d->d_cfl, c_views<T>(d, hm[m].C[cur]), hm[m].u, (int)d->n_pore, ns, vol, d->d_part,
        d->d_counter + C_MASS, d->d_scal);
    acc_total(d, hm[m].acc, d->stream, d->d_scal);
    d->timing.kernel_launches += 2;
    cudaError_t e = cudaMemcpyAsync(d->h_scal + S_OUT, d->d_scal + S_OUT,
                                    (S_OUTN - S_OUT + 1) * sizeof(double),
                                    cudaMemcpyDeviceToHost, d->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(d->stream);
    if (e != cudaSuccess) {
      s = cdi_cuda_fail(d, e, "sweep outputs");
      break;
    }
    for (int k = 0; k < ns; k++) {
      gamma[m * ns + k] = d->h_scal[S_ACC + 3 * k] * dts[m] * area;
      const double num = d->h_scal[S_OUT + 2 * k], den = d->h_scal[S_OUT + 2 * k + 1];
      const double cnt = d->h_scal[S_OUTN];
      cout[m * ns + k] = den != 0.0 ? num / den : (cnt > 0 ? d->h_scal[S_OUTP + k] / cnt : 0.0);
    }
  }
  if (s == CDI_OK) {
    cudaError_t e = cdi_timing_resolve(d);
    if (e != cudaSuccess) s = cdi_cuda_fail(d, e, "timing");
  }
  cudaStreamSynchronize(d->stream);
  if (exec) cudaGraphExecDestroy(exec);
  for (void *p : blocks) cdi_dev_release(d, p);
  return s;
}

}  // namespace

// ---------------------------------------------------------------------------
// Batch over several geometries: every (domain, combination) member in one
// launch per step.
// ---------------------------------------------------------------------------
namespace {

template <typename T, int DIM, bool PAIR, int MODE>
void launch_batch_d(cudaStream_t st, int ns, const void *members, int n, int blocks, int in) {
  const BatchMember<T> *m = (const BatchMember<T> *)members;
  switch (ns) {
    case 1: k_np_batch<T, DIM, 1, PAIR, MODE><<<blocks, kRowBlock, 0, st>>>(m, n, in); break;
    case 2: k_np_batch<T, DIM, 2, PAIR, MODE><<<blocks, kRowBlock, 0, st>>>(m, n, in); break;
    case 3: k_np_batch<T, DIM, 3, PAIR, MODE><<<blocks, kRowBlock, 0, st>>>(m, n, in); break;
    default: k_np_batch<T, DIM, 4, PAIR, MODE><<<blocks, kRowBlock, 0, st>>>(m, n, in); break;
  }
}

template <int DIM, bool PAIR>
void launch_batch32(cudaStream_t st, int ns, const void *members, int n, int blocks, int in,
                    int mode) {
  if (mode == NP_SMALL) launch_batch_d<float, DIM, PAIR, NP_SMALL>(st, ns, members, n, blocks, in);
  else if (mode == NP_LARGE) launch_batch_d<float, DIM, PAIR, NP_LARGE>(st, ns, members, n, blocks, in);
  else launch_batch_d<float, DIM, PAIR, NP_EVAL>(st, ns, members, n, blocks, in);
}

void launch_batch(const cdi_domain *lead, cudaStream_t st, const void *members, int n,
                  int blocks, int in, int mode) {
  const int ns = lead->ns;
  if (lead->prec == CDI_FP64) {
    if (lead->dim == 2) launch_batch_d<double, 2, false, NP_SMALL>(st, ns, members, n, blocks, in);
    else launch_batch_d<double, 3, false, NP_SMALL>(st, ns, members, n, blocks, in);
  } else if (lead->cpair) {
    if (lead->dim == 2) launch_batch32<2, true>(st, ns, members, n, blocks, in, mode);
    else launch_batch32<3, true>(st, ns, members, n, blocks, in, mode);
  } else {
    if (lead->dim == 2) launch_batch32<2, false>(st, ns, members, n, blocks, in, mode);
    else launch_batch32<3, false>(st, ns, members, n, blocks, in, mode);
  }
}

template <typename T>
cdi_status batch_run(cdi_domain *const *doms, int n_doms, int n_combos, int m0, int n,
                     const double *scale, const int *group, void *const *phis, const double *dts, int64_t n_steps,
                     double *gamma, double *cout) {
  cdi_domain *L = doms[0];  // the lead: its stream, allocator and scratch serve the batch
  const int ns = L->ns;
  const bool f64 = L->prec == CDI_FP64;
  std::vector<void *> blocks;
  auto take = [&](size_t bytes, bool need = true) {
    void *p = cdi_dev_alloc(L, bytes);
    for (int i = 0; i < n_doms && !p && need; i++)
      if (cdi_give_back(doms[i])) p = cdi_dev_alloc(L, bytes);
    if (p) blocks.push_back(p);
    return p;
  };
  std::vector<BatchMember<T>> hm(n);
  bool ok = true;
  int total_blocks = 0;
  for (int m = 0; m < n && ok; m++) {
    cdi_domain *d = doms[(m0 + m) / n_combos];
    const size_t TN = (size_t)d->n_pore * sizeof(T);
    void *u = take((size_t)d->dim * TN);
    const size_t CN = (size_t)ns * TN * (d->cpair ? 2 : 1);
    void *c0 = take(CN), *c1 = take(CN);
    void *acc = take((size_t)3 * kMaxSpecies * d->np_accs * 8);
    float2 *fd = f64 ? nullptr : (float2 *)take((size_t)d->dim * d->n_pore * sizeof(float2));
    if (!fd && (m == 0 || d != doms[(m0 + m - 1) / n_combos])) fd = d->d_fd;
    ok = u && c0 && c1 && acc && (f64 || fd);
    if (!ok) break;
    d->dt = dts[m];
    hm[m].s.C[0] = (T *)c0;
    hm[m].s.C[1] = (T *)c1;
    for (int in = 0; in < 2; in++)
      hm[m].s.f[in] = fields32(d, in ? c1 : c0, in ? c0 : c1, fd, nullptr, u,
                               phis[group[m]], acc);
    hm[m].s.u = (const T *)u;
    hm[m].s.phi = (const typename PhiStore<T>::type *)phis[group[m]];
    hm[m].s.acc = (typename AccSlot<T>::type *)acc;
    hm[m].s.c = make_const<T>(d);
    hm[m].g = make_geo(d);
    hm[m].block0 = total_blocks;
    hm[m].nblocks = d->np_blocks;
    total_blocks += d->np_blocks;
  }
  void *dmem = ok ? take(sizeof(BatchMember<T>) * n) : nullptr;
  int *count = dmem ? (int *)take(sizeof(int) * n) : nullptr;  // a face with |P| >= 1/2, per member
  if (!count) dmem = nullptr;
  cdi_status s = CDI_OK;
  if (!ok || !dmem) s = cdi_fail(L, CDI_ERR_OOM, "batch: device allocation failed");
  // member velocities on their domains' streams (after the lead's stream
  // has made the members' memory available: stream-ordered allocations),
  // then everything on the lead's
  if (s == CDI_OK && cudaStreamSynchronize(L->stream) != cudaSuccess)
    s = cdi_fail(L, CDI_ERR_CUDA, "batch: member memory");
  for (int m = 0; m < n && s == CDI_OK; m++)
    s = cdi_flow_scale_to(doms[(m0 + m) / n_combos], scale[m], (void *)hm[m].s.u);
  for (int i = 0; i < n_doms && s == CDI_OK; i++)
    if (cudaStreamSynchronize(doms[i]->stream) != cudaSuccess)
      s = cdi_fail(L, CDI_ERR_CUDA, "batch: member setup");
  if (s == CDI_OK && cudaMemsetAsync(count, 0, sizeof(int) * n, L->stream) != cudaSuccess)
    s = cdi_fail(L, CDI_ERR_CUDA, "batch: memset");
  for (int m = 0; m < n && s == CDI_OK; m++) {
    const cdi_domain *d = doms[(m0 + m) / n_combos];
    if (f64) {
      void *co = take(bern_bytes(d), false);
      if (co) launch_coef64(d, L->stream, hm[m].s.u, hm[m].s.phi, co);
      hm[m].s.co = (const double2 *)co;
    } else {
      member_faces(d, L->stream, hm[m].s.f, hm[m].s.u, count + m);
    }
    k_np_init<T><<<kRedBlocks, kRedThreads, 0, L->stream>>>(
        c_views<T>(d, hm[m].s.C[0]), (int)d->n_pore, ns, (T)d->c0,
        (T)(d->c0 - (double)(T)d->c0));
    L->timing.kernel_launches += 2;
    if (cudaMemsetAsync(hm[m].s.acc, 0, (size_t)3 * kMaxSpecies * d->np_accs * 8,
                        L->stream) != cudaSuccess)
      s = cdi_fail(L, CDI_ERR_CUDA, "batch: memset");
  }
  int mode = NP_SMALL;
  if (s == CDI_OK && !f64) {
    std::vector<int> large(n);
    if (cudaMemcpyAsync(large.data(), count, sizeof(int) * n, cudaMemcpyDeviceToHost,
                        L->stream) != cudaSuccess || cudaStreamSynchronize(L->stream) != cudaSuccess)
      s = cdi_fail(L, CDI_ERR_CUDA, "batch: face data");
    for (int m = 0; m < n && s == CDI_OK; m++) {
      const cdi_domain *d = doms[(m0 + m) / n_combos];
      if (large[m])
        mode = member_bern(d, L->stream, hm[m].s.f, hm[m].s.u, take(bern_bytes(d), false))
                   ? std::max<int>(mode, NP_LARGE) : NP_EVAL;
    }
  }
  if (s == CDI_OK &&
      cudaMemcpyAsync(dmem, hm.data(), sizeof(BatchMember<T>) * n, cudaMemcpyHostToDevice,
                      L->stream) != cudaSuccess)
    s = cdi_fail(L, CDI_ERR_CUDA, "batch: member table");
  cudaGraphExec_t exec = nullptr;
  int64_t done = 0;
  if (s == CDI_OK) {
    cudaEvent_t ev;
    cdi_timing_begin(L, &ev);
    if (n_steps >= kGraphSteps) {
      cudaGraph_t graph;
      cudaError_t e = cudaStreamBeginCapture(L->cap_stream, cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        for (int k = 0; k < kGraphSteps; k++)
          launch_batch(L, L->cap_stream, dmem, n, total_blocks, k & 1, mode);
        e = cudaStreamEndCapture(L->cap_stream, &graph);
      }
      if (e == cudaSuccess) {
        e = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
      }
      if (e != cudaSuccess) s = cdi_cuda_fail(L, e, "batch graph");
      while (s == CDI_OK && n_steps - done >= kGraphSteps) {
        e = cudaGraphLaunch(exec, L->stream);
        if (e != cudaSuccess) s = cdi_cuda_fail(L, e, "batch graph launch");
        done += kGraphSteps;
      }
    }
    for (; s == CDI_OK && done < n_steps; done++)
      launch_batch(L, L->stream, dmem, n, total_blocks, (int)(done & 1), mode);
    cudaError_t e = cudaGetLastError();
    if (s == CDI_OK && e != cudaSuccess) s = cdi_cuda_fail(L, e, "batch step");
    cdi_timing_end(L, ev, PH_NP, n_steps);
    L->timing.kernel_launches += n_steps;
  }
  // outputs per member, through the same reductions as a single run
  const int cur = (int)(n_steps & 1);
  for (int m = 0; m < n && s == CDI_OK; m++) {
    const cdi_domain *d = doms[(m0 + m) / n_combos];
    const double area = d->dim == 2 ? d->dx : d->dx * d->dx;
    const double vol = d->dim == 2 ? d->dx * d->dx : d->dx * d->dx * d->dx;
    k_np_sums<T><<<kRedBlocks, kRedThreads, 0, L->stream>>>(
        d->d_cfl, c_views<T>(d, hm[m].s.C[cur]), hm[m].s.u, (int)d->n_pore, ns, vol,
        L->d_part, L->d_counter + C_MASS, L->d_scal);
    acc_total(d, hm[m].s.acc, L->stream, L->d_scal);
    L->timing.kernel_launches += 2;
    cudaError_t e = cudaMemcpyAsync(L->h_scal + S_OUT, L->d_scal + S_OUT,
                                    (S_OUTN - S_OUT + 1) * sizeof(double),
                                    cudaMemcpyDeviceToHost, L->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(L->stream);
    if (e != cudaSuccess) {
      s = cdi_cuda_fail(L, e, "batch outputs");
      break;
    }
    for (int k = 0; k < ns; k++) {
      gamma[m * ns + k] = L->h_scal[S_ACC + 3 * k] * dts[m] * area;
      const double num = L->h_scal[S_OUT + 2 * k], den = L->h_scal[S_OUT + 2 * k + 1];
      const double cnt = L->h_scal[S_OUTN];
      cout[m * ns + k] = den != 0.0 ? num / den : (cnt > 0 ? L->h_scal[S_OUTP + k] / cnt : 0.0);
    }
  }
  if (s == CDI_OK) {
    cudaError_t e = cdi_timing_resolve(L);
    if (e != cudaSuccess) s = cdi_cuda_fail(L, e, "timing");
  }
  cudaStreamSynchronize(L->stream);
  if (exec) cudaGraphExecDestroy(exec);
  for (void *p : blocks) cdi_dev_release(L, p);
  return s;
}

}  // namespace

// Members [m, m + n) by run(m, n), in halves where their memory cannot be had
// at once (members are independent: the same bits).
template <typename R> static cdi_status in_parts(int m, int n, const R &run) {
  cdi_status s = run(m, n);
  if (s != CDI_ERR_OOM || n < 2) return s;
  s = in_parts(m, n / 2, run);
  return s == CDI_OK ? in_parts(m + n / 2, n - n / 2, run) : s;
}

cdi_status cdi_np_batch(cdi_domain *const *doms, int n_doms, int n_combos, const double *scale,
                        const int *group, void *const *phis, const double *dts, int64_t n_steps,
                        double *gamma, double *cout) {
  const int ns = doms[0]->ns;
  return in_parts(0, n_doms * n_combos, [&](int m, int n) {
    auto *run = doms[0]->prec == CDI_FP64 ? batch_run<double> : batch_run<float>;
    return run(doms, n_doms, n_combos, m, n, scale + m, group + m, phis, dts + m, n_steps,
               gamma + (size_t)m * ns, cout + (size_t)m * ns);
  });
}

cdi_status cdi_np_sweep(cdi_domain *d, int n_members, const double *scale, const int *group,
                        void *const *phi_groups, const double *dts, int64_t n_steps,
                        double *gamma, double *cout) {
  return in_parts(0, n_members, [&](int m, int n) {
    auto *run = d->prec == CDI_FP64 ? sweep_run<double> : sweep_run<float>;
    return run(d, n, scale + m, group + m, phi_groups, dts + m, n_steps,
               gamma + (size_t)m * d->ns, cout + (size_t)m * d->ns);
  });
}

// Coupled stepping (Eq. 3-5): before every block of couple_K steps (counted
// from cdi_init_transport) the potential is re-solved from the current
// concentrations; the steps of a block are plain launches.
static cdi_status np_steps_coupled(cdi_domain *d, int64_t n) {
  const int64_t K = d->couple_K;
  while (n > 0) {
    if (d->np_steps % K == 0) {
      cdi_status s = cdi_psi_coupled(d);
      if (s != CDI_OK) return s;
    }
    const int64_t block = std::min<int64_t>(n, K - d->np_steps % K);
    if (d->imp_tol > 0.0) {  // implicit steps in the re-solved potential
      cdi_status s = cdi_imp_steps(d, block);
      if (s != CDI_OK) return s;
      n -= block;
      continue;
    }
    if (d->faces_stale) {
      cdi_status s = cdi_np_faces(d);
      if (s != CDI_OK) return s;
    }
    cudaEvent_t ev;
    cdi_timing_begin(d, &ev);
    for (int64_t k = 0; k < block; k++) {
      launch_step(d, d->stream, d->cur, k > 0);
      d->cur = 1 - d->cur;
    }
    CDI_TRY(d, cudaGetLastError(), "transport step");
    cdi_timing_end(d, ev, PH_NP, block);
    d->timing.kernel_launches += block;
    d->np_steps += block;
    n -= block;
  }
  return CDI_OK;
}

cdi_status cdi_np_steps(cdi_domain *d, int64_t n) {
  if (n == 0) return CDI_OK;
  if (d->couple_K > 0) return np_steps_coupled(d, n);
  if (d->imp_tol > 0.0) return cdi_imp_steps(d, n);
  if (d->faces_stale) {
    cdi_status s = cdi_np_faces(d);
    if (s != CDI_OK) return s;
  }
  cudaEvent_t ev;
  cdi_timing_begin(d, &ev);
  int64_t left = n;
  if (d->cur == 1) {
    launch_step(d, d->stream, 1, false);
    d->cur = 0;
    left--;
  }
  if (left >= kGraphSteps) {
    if (!d->np_graph) {
      cudaGraph_t graph;
      CDI_TRY(d, cudaStreamBeginCapture(d->cap_stream, cudaStreamCaptureModeThreadLocal),
              "begin capture");
      for (int k = 0; k < kGraphSteps; k++) launch_step(d, d->cap_stream, k & 1, k > 0);
      cudaError_t e = cudaStreamEndCapture(d->cap_stream, &graph);
      CDI_TRY(d, e, "end capture");
      e = cudaGraphInstantiate(&d->np_graph, graph, 0);
      cudaGraphDestroy(graph);
      CDI_TRY(d, e, "instantiate transport graph");
    }
    while (left >= kGraphSteps) {
      CDI_TRY(d, cudaGraphLaunch(d->np_graph, d->stream), "transport graph");
      left -= kGraphSteps;
    }
  }
  for (bool dep = false; left > 0; left--, dep = true) {
    launch_step(d, d->stream, d->cur, dep);
    d->cur = 1 - d->cur;
  }
  CDI_TRY(d, cudaGetLastError(), "transport step");
  cdi_timing_end(d, ev, PH_NP, n);
  d->timing.kernel_launches += n;
  d->np_steps += n;
  return CDI_OK;
}

cdi_status cdi_np_reduce(cdi_domain *d) {
  const double vol = d->dim == 2 ? d->dx * d->dx : d->dx * d->dx * d->dx;
  if (d->prec == CDI_FP64)
    k_np_sums<double><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        d->d_cfl, c_views<double>(d, d->d_C[d->cur]), (const double *)d->d_u,
        (int)d->n_pore, d->ns, vol, d->d_part, d->d_counter + C_MASS, d->d_scal);
  else
    k_np_sums<float><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        d->d_cfl, c_views<float>(d, d->d_C[d->cur]), (const float *)d->d_u,
        (int)d->n_pore, d->ns, vol, d->d_part, d->d_counter + C_MASS, d->d_scal);
  acc_total(d, d->d_acc, d->stream, d->d_scal);
  d->timing.kernel_launches += 2;
  CDI_TRY(d, cudaGetLastError(), "transport sums");
  CDI_TRY(d, cudaMemcpyAsync(d->h_scal + S_OUT, d->d_scal + S_OUT,
                             (S_OUTN - S_OUT + 1) * sizeof(double), cudaMemcpyDeviceToHost,
                             d->stream),
          "sums copy");
  CDI_TRY(d, cudaStreamSynchronize(d->stream), "transport sums");
  CDI_TRY(d, cdi_timing_resolve(d), "timing");
  return CDI_OK;
}

cdi_status cdi_np_geometry(cdi_domain *d, double *pores, double *faces, double *sum_ux) {
  if (d->prec == CDI_FP64)
    k_geometry<double><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        d->d_cfl, (const double *)d->d_u, (int)d->n_pore, 2 * d->dim, d->d_part,
        d->d_counter + C_GEOM, d->d_scal);
  else
    k_geometry<float><<<kRedBlocks, kRedThreads, 0, d->stream>>>(
        d->d_cfl, (const float *)d->d_u, (int)d->n_pore, 2 * d->dim, d->d_part,
        d->d_counter + C_GEOM, d->d_scal);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "geometry");
  CDI_TRY(d, cudaMemcpyAsync(d->h_scal + S_GEOM, d->d_scal + S_GEOM, 3 * sizeof(double),
                             cudaMemcpyDeviceToHost, d->stream),
          "geometry copy");
  CDI_TRY(d, cudaStreamSynchronize(d->stream), "geometry");
  *pores = d->h_scal[S_GEOM];
  *faces = d->h_scal[S_GEOM + 1];
  if (sum_ux) *sum_ux = d->h_scal[S_GEOM + 2];
  return CDI_OK;
}

cdi_status cdi_np_column_means(cdi_domain *d, int k) {
  const int rows = d->ny * d->nz;
  if (d->prec == CDI_FP64)
    k_colmeans<double><<<d->nx, kRedThreads, 0, d->stream>>>(
        d->d_words, d->W, c_view<double>(d, d->d_C[d->cur], k), rows, d->d_colout);
  else
    k_colmeans<float><<<d->nx, kRedThreads, 0, d->stream>>>(
        d->d_words, d->W, c_view<float>(d, d->d_C[d->cur], k), rows, d->d_colout);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "column means");
  return CDI_OK;
}

// Face flags, row words and lateral links of the compact transport layout (after the
// pore lists and the face flags).
cdi_status cdi_np_build_compact(cdi_domain *d) {
  const int n = (int)d->n_pore;
  const long long n_words = (long long)d->ny * d->nz * d->W;
  k_cfl<<<kRedBlocks, kRedThreads, 0, d->stream>>>(d->d_nflags, d->d_cell_list, n, d->d_cfl);
  k_words<<<kRedBlocks, kRedThreads, 0, d->stream>>>(d->d_nflags, d->d_cell_list, n, d->nx, d->W,
                                                     n_words, d->d_words);
  k_lat_nbr<<<kRedBlocks, kRedThreads, 0, d->stream>>>(d->d_cfl, d->d_cell_list, d->d_words, n,
                                                       d->nx, d->W, d->ny, d->nz, d->walls,
                                                       2 * d->dim, d->d_latnb);
  if (d->dim == 2)
    k_lat_pack<2><<<kRedBlocks, kRedThreads, 0, d->stream>>>(d->d_latnb, n, d->d_latd, d->d_latb);
  else
    k_lat_pack<3><<<kRedBlocks, kRedThreads, 0, d->stream>>>(d->d_latnb, n, d->d_latd, d->d_latb);
  d->timing.kernel_launches += 4;
  CDI_TRY(d, cudaGetLastError(), "compact layout");
  return CDI_OK;
}

// Rank-ordered fields of the domain's precision (species k of the current
// concentrations, or with species < 0 the dim velocity components) -> FP64
// lattice fields (dst: N doubles each, 0 in solid cells).
template <typename T> static void scatter(cdi_domain *d, int species, double *dst) {
  CViews<T> v{};
  int comps = 1;
  if (species >= 0) {
    v.v[0] = c_view<T>(d, d->d_C[d->cur], species);
  } else {
    comps = d->dim;
    for (int a = 0; a < comps; a++)
      v.v[a] = CView<T>{(const T *)d->d_u + (size_t)a * d->n_pore, 1, 0};
  }
  k_scatter<T><<<kRedBlocks, kRedThreads, 0, d->stream>>>(v, comps, d->d_cell_list,
                                                          (int)d->n_pore, d->N, dst);
}
cdi_status cdi_np_scatter(cdi_domain *d, int species, double *dst) {
  const int comps = species >= 0 ? 1 : d->dim;
  CDI_TRY(d, cudaMemsetAsync(dst, 0, (size_t)comps * d->N * 8, d->stream), "scatter reset");
  if (d->prec == CDI_FP64) scatter<double>(d, species, dst);
  else scatter<float>(d, species, dst);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "scatter");
  return CDI_OK;
}

// FP32 concentrations of buffer b as the planes of a saved state, and back.
cdi_status cdi_np_records_to_planes(cdi_domain *d, int b, float *planes) {
  const size_t np = (size_t)kMaxSpecies * d->n_pore;
  k_records_to_planes<<<kRedBlocks, kRedThreads, 0, d->stream>>>(
      c_views<float>(d, d->d_C[b]), (int)d->n_pore, d->ns, planes, d->cpair ? planes + np : nullptr);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "state planes");
  return CDI_OK;
}
cdi_status cdi_np_planes_to_records(cdi_domain *d, const float *planes, int b) {
  const size_t np = (size_t)kMaxSpecies * d->n_pore;
  k_planes_to_records<<<kRedBlocks, kRedThreads, 0, d->stream>>>(
      c_views<float>(d, d->d_C[b]), (int)d->n_pore, d->ns, planes, d->cpair ? planes + np : nullptr);
  d->timing.kernel_launches++;
  CDI_TRY(d, cudaGetLastError(), "state planes");
  return CDI_OK;
}
