// Internal declarations of the GB300 CDI library: the domain object, device
// helpers shared by the kernels, and the lattice tables.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/cdi.h"

namespace cdi {

constexpr int kMaxSpecies = 4;
constexpr int kRowBlock = 128;      // threads per block along x for stencils
constexpr int kRedThreads = 256;    // threads per block for reductions
constexpr int kRedBlocks = 4 * 152; // fixed grid of the grid-stride reductions

// ---------------------------------------------------------------------------
// Lattices (D2Q9 and D3Q19 of Sec. 2).  Direction i and its opposite are
// paired as i <-> i + (Q-1)/2 so that opp() is arithmetic.
// ---------------------------------------------------------------------------
template <int DIM> struct Lat;

template <> struct Lat<2> {
  static constexpr int Q = 9;
  static constexpr int H = 4;
  __host__ __device__ static constexpr int ex(int i) {
    return i == 1 || i == 3 || i == 8 ? 1 : (i == 4 || i == 5 || i == 7 ? -1 : 0);
  }
  __host__ __device__ static constexpr int ey(int i) {
    return i == 2 || i == 3 || i == 4 ? 1 : (i == 6 || i == 7 || i == 8 ? -1 : 0);
  }
  __host__ __device__ static constexpr int ez(int) { return 0; }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 4.0 / 9.0 : ((ex(i) * ex(i) + ey(i) * ey(i)) == 1 ? 1.0 / 9.0 : 1.0 / 36.0);
  }
  __host__ __device__ static constexpr int opp(int i) {
    return i == 0 ? 0 : (i <= H ? i + H : i - H);
  }
};

template <> struct Lat<3> {
  static constexpr int Q = 19;
  static constexpr int H = 9;
  // 1:(1,0,0) 2:(0,1,0) 3:(0,0,1) 4:(1,1,0) 5:(1,-1,0) 6:(1,0,1) 7:(1,0,-1)
  // 8:(0,1,1) 9:(0,1,-1); 10..18 are their negatives.
  __host__ __device__ static constexpr int bx(int k) {
    return k == 1 || k == 4 || k == 5 || k == 6 || k == 7 ? 1 : 0;
  }
  __host__ __device__ static constexpr int by(int k) {
    return k == 2 || k == 4 || k == 8 || k == 9 ? 1 : (k == 5 ? -1 : 0);
  }
  __host__ __device__ static constexpr int bz(int k) {
    return k == 3 || k == 6 || k == 8 ? 1 : (k == 7 || k == 9 ? -1 : 0);
  }
  __host__ __device__ static constexpr int ex(int i) {
    return i == 0 ? 0 : (i <= H ? bx(i) : -bx(i - H));
  }
  __host__ __device__ static constexpr int ey(int i) {
    return i == 0 ? 0 : (i <= H ? by(i) : -by(i - H));
  }
  __host__ __device__ static constexpr int ez(int i) {
    return i == 0 ? 0 : (i <= H ? bz(i) : -bz(i - H));
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 1.0 / 3.0
                  : ((ex(i) * ex(i) + ey(i) * ey(i) + ez(i) * ez(i)) == 1 ? 1.0 / 18.0
                                                                         : 1.0 / 36.0);
  }
  __host__ __device__ static constexpr int opp(int i) {
    return i == 0 ? 0 : (i <= H ? i + H : i - H);
  }
};

// Flow-site flag word: bit 0 = the site is solid; bit i (1..Q-1) = the
// neighbour along e_i is solid or lies beyond a lateral wall; bits Q..Q+5 =
// the site lies on the high/low x, y, z edge of the flow grid, where the
// periodic neighbour offsets wrap around.
template <int DIM> struct FlowFlag;
template <> struct FlowFlag<2> { using type = uint16_t; };
template <> struct FlowFlag<3> { using type = uint32_t; };
template <int DIM> struct WrapBit {
  static constexpr int XHI = Lat<DIM>::Q, XLO = XHI + 1, YHI = XHI + 2, YLO = XHI + 3,
                       ZHI = XHI + 4, ZLO = XHI + 5;
};

// Transport-cell flag word: bit 0 = solid; bit 1 + f = the neighbour across
// face f (f = +x,-x,+y,-y,+z,-z) is a solid voxel inside the image (after the
// periodic wrap); bit 7 + f = face f lies on the image boundary.
using NFlag = uint16_t;
constexpr int kFaceBit = 1;
constexpr int kEdgeBit = 7;

// 16-bit lateral differences: a closed face, and one that does not fit.
constexpr short kLatClosed = -32768, kLatWide = -32767;

// ---------------------------------------------------------------------------
// Deterministic block reductions (fixed order, no floating-point atomics).
// ---------------------------------------------------------------------------
template <int NV, typename V, typename Op>
__device__ __forceinline__ void warp_reduce(V (&v)[NV], Op op) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] = op(v[k], __shfl_down_sync(0xffffffffu, v[k], o));
}

struct OpSum {
  template <typename V> __device__ V operator()(V a, V b) const { return a + b; }
};
struct OpMax {
  template <typename V> __device__ V operator()(V a, V b) const { return a > b ? a : b; }
};

// Reduces v over the block; the result is valid in thread 0.  smem must hold
// NV * 32 values.  All threads of the block must call it.
template <int NV, typename V, typename Op>
__device__ __forceinline__ void block_reduce(V (&v)[NV], V *smem, Op op, V identity) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
  warp_reduce<NV>(v, op);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < NV; k++) smem[k * 32 + w] = v[k];
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] = lane < nw ? smem[k * 32 + lane] : identity;
    warp_reduce<NV>(v, op);
  }
  __syncthreads();
}

// Called by every thread after the block wrote its partials: returns true in
// the last block to finish (which then combines all partials in a fixed
// order and must reset *counter to 0).
__device__ __forceinline__ bool last_block(unsigned int *counter, int nblocks) {
  __shared__ bool am_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) am_last = (atomicAdd(counter, 1u) == (unsigned)(nblocks - 1));
  __syncthreads();
  return am_last;
}

// Sums partials[k * nblocks + b] over b for each k (fixed order) in the last
// block; the result lands in thread 0's v.
template <int NV, typename Op>
__device__ __forceinline__ void combine_partials(const double *partials, int nblocks,
                                                 double (&v)[NV], double *smem, Op op,
                                                 double identity) {
#pragma unroll
  for (int k = 0; k < NV; k++) v[k] = identity;
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] = op(v[k], __ldcg(partials + (size_t)k * nblocks + b));
  block_reduce<NV>(v, smem, op, identity);
}

// ---------------------------------------------------------------------------
// Programmatic dependent launch: a kernel launched by launch_pdl with early
// set may start while the kernel before it in the stream (or captured graph)
// still runs, as soon as all blocks of that kernel have called pdl_launch or
// ended.
// pdl_wait returns once that kernel has ended and its writes are visible;
// before it only data that no kernel of the sequence writes may be read, and
// nothing written.  Data that the sequence writes is read by plain loads (not
// through the non-coherent path, whose loads may be moved).  It takes the gap
// between steps, 0.5 to 2 us: device time of a step without and with it, 128x64
// FP64 flow 3.4 and 2.8 us, transport 4.1 and 3.2; 1024x512 pair flow 11.9 and
// 11.4, transport 6.0 and 5.1; transport of a resolved 101x87x93 pack 13.9 and
// 13.0; 256^3 flow 438.4 and 437.4, transport 140.5 and 138.1.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
void launch_pdl(void (*kernel)(P...), dim3 grid, int threads, cudaStream_t st, bool early,
                A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = early ? 1 : 0;
  (void)cudaLaunchKernelEx(&cfg, kernel, P(args)...);  // (callers read cudaGetLastError)
}

// ---------------------------------------------------------------------------
// Iterative solvers as one cooperative launch: one block an SM, every vector
// pass a grid-stride loop, the passes separated by grid barriers that carry
// the dot products of all systems at once.
//
// A barrier's cost is a chain of latencies, so its sums run side by side: each
// value has its own warps in the block and its own warp over the blocks'
// partials.  FP64 values go through shared memory (a shuffle tree in every
// warp costs five FP64 instructions a value at 2 lanes an SM), their additions
// as few deep as a tree allows (each takes some 0.1 us of latency); FP32 (sum,
// error) pairs stay pairs up to the total.  152 blocks of 1024
// threads: 1.6 us without sums, 5.3 us with two FP64 sums (6.0 added in a
// row), 3.9 us with two pairs.
// ---------------------------------------------------------------------------
constexpr int kGridThreads = 1024;
constexpr long long kBarrierPolls = 1ll << 26;  // tens of seconds
constexpr int kGridSums = 2 * kMaxSpecies;      // dot products of a phase, at most

struct GridBarrier {
  unsigned *counter;  // arrivals since the launch (0 before it)
  double *part;       // 2 * kGridSums * gridDim.x partials
  double *sm;         // shared: a row of values per sum, then kGridSums * 8
  int row;            // values of a row: blockDim.x (FP64) or one a warp (FP32)
  unsigned target;
  int parity;         // which half of part this phase writes: a block may be
                      // reading the last phase's half still
};

// A thread's contribution to sum k of the phase (row = blockDim.x), or its
// warp's from every lane's (sum, error) pair (row = blockDim.x / 32).
__device__ __forceinline__ void grid_add(const GridBarrier &b, int k, double v) {
  b.sm[k * b.row + threadIdx.x] = v;
}
__device__ __forceinline__ float2 pair_sum(float2 a, float2 b) {
  const float u = __fadd_rn(a.x, b.x), w = __fsub_rn(u, a.x);
  const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(u, w)), __fsub_rn(b.x, w));
  return make_float2(u, __fadd_rn(__fadd_rn(a.y, b.y), e));
}
__device__ __forceinline__ double pair_sum(double a, double b) { return a + b; }
__device__ __forceinline__ float2 warp_sum(float2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = pair_sum(v, make_float2(__shfl_down_sync(0xffffffffu, v.x, o),
                                __shfl_down_sync(0xffffffffu, v.y, o)));
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ void grid_add(const GridBarrier &b, int k, float s, float c) {
  const float2 v = warp_sum(make_float2(s, c));
  if ((threadIdx.x & 31) == 0)
    reinterpret_cast<float2 *>(b.sm)[k * b.row + (threadIdx.x >> 5)] = v;
}

// Barrier over the grid (whose blocks are all resident: a cooperative launch)
// and this phase's nv sums in tot[0 .. nv), in a fixed order and the same bits
// in every block; V is double, or float2 for (sum, error) pairs.  False in
// every thread of a block whose wait ran into its limit: the block must return
// (the others then run into theirs).
template <typename V>
__device__ __forceinline__ bool grid_totals(GridBarrier &b, V *tot, int nv) {
  static_assert(sizeof(V) == 8, "a sum is 8 bytes");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  V *sm = reinterpret_cast<V *>(b.sm), *red = sm + nv * b.row;
  V *part = reinterpret_cast<V *>(b.part) + (size_t)b.parity * kGridSums * gridDim.x;
  const V zero{};
  // warps that share a sum: a power of two, at most 8 and no more than its row fills
  int share = 1;
  while (2 * share * max(nv, 1) <= warps && 2 * share * 32 <= b.row && share < 8) share *= 2;
  __syncthreads();
  for (int k = warp / share; k < nv; k += warps / share) {
    const V *v = sm + k * b.row;
    const int step = 32 * share, j = (warp % share) * 32 + lane;
    V s[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      s[u] = j + u * step < b.row ? v[j + u * step] : zero;
      for (int i = j + (u + 4) * step; i < b.row; i += 4 * step) s[u] = pair_sum(s[u], v[i]);
    }
    const V t = warp_sum(pair_sum(pair_sum(s[0], s[1]), pair_sum(s[2], s[3])));
    if (lane == 0) red[k * 8 + warp % share] = t;
  }
  if (nv) __syncthreads();
  b.target += gridDim.x;
  int ok = 1;
  if (warp == 0) {
    if (lane < nv) {
      V s[8];
#pragma unroll
      for (int u = 0; u < 8; u++) s[u] = u < share ? red[lane * 8 + u] : zero;
#pragma unroll
      for (int h = 4; h > 0; h >>= 1)
#pragma unroll
        for (int u = 0; u < h; u++)
          if (u + h < share) s[u] = pair_sum(s[u], s[u + h]);
      __stcg(part + (size_t)lane * gridDim.x + blockIdx.x, s[0]);
    }
    __syncwarp();
    if (lane == 0) {
      // the arrival releases the block's writes (which the barrier above put
      // before it), the fence behind the last look acquires the other blocks'
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(b.counter) : "memory");
      ok = 0;
      for (long long i = 0; i < kBarrierPolls && !ok; i++) {
        unsigned c;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(b.counter) : "memory");
        ok = (int)(c - b.target) >= 0;
      }
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
    }
  }
  if (!__syncthreads_and(ok)) return false;
  b.parity ^= 1;
  if (nv == 0) return true;
  for (int k = warp; k < nv; k += warps) {
    const V *p = part + (size_t)k * gridDim.x;
    const int G = (int)gridDim.x;
    V s[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      s[u] = lane + 32 * u < G ? __ldcg(p + lane + 32 * u) : zero;
      for (int i = lane + 32 * (u + 4); i < G; i += 128) s[u] = pair_sum(s[u], __ldcg(p + i));
    }
    const V t = warp_sum(pair_sum(pair_sum(s[0], s[1]), pair_sum(s[2], s[3])));
    if (lane == 0) tot[k] = t;
  }
  __syncthreads();
  return true;
}
__device__ __forceinline__ void grid_give_up(double *flag) {
  if (threadIdx.x == 0) *flag = 1.0;
}
// Shared bytes of a GridBarrier with nv rows.
inline size_t grid_smem(int threads, int row_div, int nv) {
  return ((size_t)nv * (threads / row_div) + kGridSums * 8) * sizeof(double);
}

// Blocks and threads of a cooperative launch over n items: one block an SM,
// as few threads as cover the items (few items are spread over all SMs, whose
// FP64 units are the bound); smem is a thread's share of the shared memory.
// 0 if not even one block fits.
int grid_shape(const void *kernel, long long n, int row_div, int nv, int *threads, size_t *smem);

// psi / V_T as stored for the transport kernel: FP64, or an unevaluated
// FP32 pair hi + lo (so that face differences keep FP64-like accuracy while
// the arithmetic stays on the FP32 units).
template <typename T> struct PhiStore;
template <> struct PhiStore<double> {
  using type = double;
  __device__ static double make(double v) { return v; }
  __device__ static double zero() { return 0.0; }
};
template <> struct PhiStore<float> {
  using type = float2;
  __device__ static float2 make(double v) {
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (double)hi));
  }
  __device__ static float2 zero() { return make_float2(0.f, 0.f); }
};

// Arithmetic with explicit rounding (never contracted into FMAs by the
// compiler, so two kernels that inline the same function compute the same
// bits).
__device__ __forceinline__ double r_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double r_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double r_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double r_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float r_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float r_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float r_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float r_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// Bernoulli function pair B(x), B(-x) with B(x) = x / (exp(x) - 1), from one
// expm1 of |x|: B(|x|) directly (series near 0) and B(-|x|) = B(|x|) + |x|,
// both positive so neither loses precision.
template <typename T>
__device__ __forceinline__ void bernoulli_pair(T x, T &Bx, T &Bmx) {
  const T a = fabs(x);
  T Ba;
  if (a < T(1e-3)) {
    // 1 - a/2 + a^2/12 - a^4/720
    const T a2 = r_mul(a, a);
    Ba = r_fma(a2, r_fma(a2, T(-1) / T(720), T(1) / T(12)), r_fma(a, T(-0.5), T(1)));
  } else {
    Ba = a / expm1(a);
  }
  const T Bma = r_add(Ba, a);
  if (x >= T(0)) {
    Bx = Ba;
    Bmx = Bma;
  } else {
    Bx = Bma;
    Bmx = Ba;
  }
}

}  // namespace cdi

// ---------------------------------------------------------------------------
// The domain object behind the opaque handle.
// ---------------------------------------------------------------------------
struct cdi_domain {
  // geometry
  int dim = 2, nx = 0, ny = 0, nz = 1, walls = 0, mirror = 1, prec = CDI_FP64;
  double dx = 1e-7;
  int NX = 0;         // flow-grid extent along x (2 nx with the mirror)
  long long N = 0;    // transport cells nx*ny*nz
  long long Nf = 0;   // flow sites NX*ny*nz
  long long n_pore = 0, n_pore_inlet = 0;
  uint64_t mask_hash = 0;  // FNV-1a of the mask bytes (identifies a saved state's geometry)

  // execution
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  cudaStream_t cap_stream = nullptr;  // private stream used only for capture
  cdi_allocator alloc{};
  bool has_alloc = false;
  std::string err;
  struct Block {
    void *p;       // what cdi_dev_alloc returned
    size_t bytes;
    void *base;    // what the allocator returned
  };
  std::vector<Block> blocks;

  // device buffers
  uint8_t *d_mask = nullptr;    // N
  cdi::NFlag *d_nflags = nullptr;  // N face flags
  int *d_flow_list = nullptr;   // pore sites of the flow grid, ascending
  long long n_flow_pore = 0;
  // neighbour data of the odd LBM step (see flow.cu): per pore rank a flag
  // word and one signed byte per lateral row offset (the offset's rank base
  // less the rank and the base of the rank's 32-rank tile); per tile the
  // bases; full neighbour ranks of the x-edge sites and of the sites whose
  // bytes overflow in a table of n_lovf = 2 ny nz + (those sites) slots
  unsigned *d_lf = nullptr;     // n_flow_pore
  unsigned *d_ld = nullptr;     // (1 in 2D, 2 in 3D) words * n_flow_pore
  int *d_lb = nullptr;          // (2 in 2D, 8 in 3D) * n_ltiles
  int n_ltiles = 0;             // ceil(n_flow_pore / 32)
  int *d_lovf = nullptr;        // (Q-1) * n_lovf
  int n_lovf = 0;
  int *d_cell_list = nullptr;   // pore cells of the transport grid, ascending:
                                // entry r is the lattice cell of pore rank r
  cdi::NFlag *d_cfl = nullptr;  // n_pore: face flags
  uint2 *d_words = nullptr;     // ny*nz*W: per 32 cells of a row {rank of the
                                // first pore cell at or after it, pore bits}
  int W = 0;                    // words per row, ceil(nx / 32)
  int *d_latnb = nullptr;       // 2*(dim-1)*n_pore lateral neighbour ranks (-1: none)
  void *d_g = nullptr;          // Q*n_flow_pore populations (shifted) by pore rank
  float *d_glo = nullptr;       // their low parts (pair storage only)
  double *d_uflow = nullptr;    // dim*Nf lattice velocity (last check), FP64
  // transport fields by pore rank (component a / species k of rank r at
  // a * n_pore + r)
  void *d_u = nullptr;          // dim*n_pore scaled velocity, precision T
  double *d_psi = nullptr;      // N potential (V), FP64, lattice order
  void *d_phi = nullptr;        // n_pore psi / V_T, 8 bytes a cell: double
                                // (FP64) or a float2 (hi, lo) pair (FP32)
  bool cpair = false;           // concentrations stored as FP32 pairs (hi + lo)
  void *d_C[2] = {nullptr, nullptr};  // concentrations, ping-pong.  FP64: species
                                // k of rank r at k * n_pore + r.  FP32: one record
                                // per rank and species pair (2p, 2p + 1), the pairs
                                // one after the other: c_2p[, c_2p+1][, their low
                                // words] (see c_view); the layout follows ns
  float2 *d_fd = nullptr;       // FP32: dim * n_pore face data (see k_np_faces)
  void *d_bern = nullptr;       // FP32: Bernoulli pairs of the faces with |P| >= 1/2
                                // (taken the first time there is one); FP64: face
                                // coefficients (taken for the first explicit steps);
                                // done without where memory is short
  size_t bern_bytes = 0;
  int np_mode = 0;              // which kernel the faces ask for (see np_warp31)
  bool faces_stale = true;      // d_fd, d_bern and np_mode are not those of the
                                // current potential (explicit steps form them again)
  short *d_latd = nullptr;      // 2*(dim-1) 16-bit lateral differences per rank
  int *d_latb = nullptr;        // and their bases per tile of 31 ranks
  double *d_acc = nullptr;      // 3*kMaxSpecies*np_accs per-warp sums (8 B each:
                                // FP64, or an FP32 pair in FP32 modes)
  double *d_part = nullptr;     // reduction partials (8*kRedBlocks)
  unsigned int *d_counter = nullptr;  // last-block counters (8 slots)
  double *d_scal = nullptr;     // device scalars (S_COUNT)
  double *h_scal = nullptr;     // pinned host copy of the scalars (S_COUNT)
  double *d_cg = nullptr;       // 4*N CG work vectors (r, p, q, diag), scratch of
                                // other calls between solves
  double *d_colout = nullptr;   // nx column means

  // state
  bool flow_done = false, psi_done = false, np_ready = false;
  int64_t flow_steps = 0;
  double flow_residual = 0.0;
  double U_lat = 0.0;           // pore-mean lattice x velocity
  double U_target = 0.0;
  double tau = 1.0, force = 0.0;
  int ns = 0;
  int z[cdi::kMaxSpecies] = {0, 0, 0, 0};
  double D[cdi::kMaxSpecies] = {0, 0, 0, 0};
  double c0 = 0.0, Ka = 0.0, dt = 0.0, VT = 0.0;
  // potential parameters of the last cdi_set_potential (for the coupled
  // re-solve) and the coupling period (0: frozen potential)
  double psi_s = 0.0, eps_r = 78.5, psi_tol = 1e-12;
  int psi_max_iter = 100000;
  int64_t couple_K = 0;
  // implicit (backward Euler) transport: on when imp_tol > 0
  double imp_tol = 0.0;
  int imp_max_iter = 0;
  bool imp_stale = true;        // the operator must be rebuilt before a step
  int64_t imp_iters = 0;        // linear iterations so far
  double imp_last_rel = 0.0;    // last relative residual
  double *d_icoef = nullptr;    // operator coefficients of every species (FP64)
  double *d_iwork = nullptr;    // imp_sets * 5 * n_pore FP64 work vectors
  int imp_sets = 0;             // species whose vectors d_iwork holds
  double *d_iscal = nullptr;    // the solver's device scalars (16)
  double *d_src = nullptr;      // N charge terms of Eq. 4 (coupled mode only)
  int cur = 0;                  // which of d_C holds the current state
  int64_t np_steps = 0;
  int np_blocks = 0;            // 128-thread blocks of the fused sweep/batch
                                // steps (FP64: one thread per pore cell; FP32:
                                // warps of 31 home cells)
  int np_accs = 0;              // account sets, one per warp (rounded up to a
                                // multiple of 8: enough for any launch shape)
  // block sizes of the step kernels
  int lbm_block = 128, np_block = 128;
  int np_variant = 1;           // transport launch shape (see kNpVariantBlock)
  int lbm_variant = 1;          // LBM launch shape (see tune_lbm)
  bool lbm_tuned = false, np_tuned = false;

  // graphs
  cudaGraphExec_t flow_graph = nullptr;
  int flow_graph_K = 0;
  double flow_graph_tau = 0.0, flow_graph_force = 0.0;
  cudaGraphExec_t np_graph = nullptr;
  int np_graph_steps = 0;

  // timing
  struct EvPair {
    cudaEvent_t a, b;
    int phase;
    int64_t launches;
  };
  std::vector<EvPair> pending;
  std::vector<cudaEvent_t> ev_pool;
  cdi_timing timing{};
};

namespace cdi {

// One species of a concentration buffer: hi word of rank r at p[r * stride],
// its low word (pair storage; lo != 0) lo words further on.
template <typename T> struct CView {
  const T *p;
  int stride, lo;
  __device__ __forceinline__ double at(int r) const {
    const T *q = p + (size_t)r * stride;
    return (double)q[0] + (lo ? (double)q[lo] : 0.0);
  }
};
template <typename T> struct CViews {
  CView<T> v[kMaxSpecies];
};
template <typename T> inline CView<T> c_view(const cdi_domain *d, const void *C, int k) {
  if (sizeof(T) == 8) return CView<T>{(const T *)C + (size_t)k * d->n_pore, 1, 0};
  const int per = d->cpair ? 2 : 1, pair = k / 2, w = d->ns - 2 * pair >= 2 ? 2 : 1;
  return CView<T>{(const T *)C + (size_t)pair * 2 * per * d->n_pore + (k & 1), w * per,
                  d->cpair ? w : 0};
}
template <typename T> inline CViews<T> c_views(const cdi_domain *d, const void *C) {
  CViews<T> v{};
  for (int k = 0; k < d->ns; k++) v.v[k] = c_view<T>(d, C, k);
  return v;
}

}  // namespace cdi

// Scalar slots in d_scal / h_scal.
enum {
  S_RES_NUM = 0, S_RES_DEN = 1, S_RES = 2,  // flow residual
  S_ULAT = 3, S_SCALE = 4,                  // velocity export
  S_CG_RZ = 8, S_CG_PQ = 9, S_CG_ALPHA = 10, S_CG_BETA = 11, S_CG_RR = 12,
  S_CG_BB = 13, S_CG_REL = 14, S_CG_DONE = 15, S_CG_TOL = 16, S_CG_IT = 17,
  S_PB_FF = 18, S_PB_BB = 19,               // Poisson-Boltzmann Newton residual
  S_RATE = 20, S_DT = 21,                   // time step
  S_OUT = 24,                               // 2*kMaxSpecies: outlet sums
  S_MASS = 32,                              // kMaxSpecies
  S_OUTP = 36,                              // kMaxSpecies: plain outlet sums
  S_ACC = 40,                               // 3*kMaxSpecies: Gamma/In/Out sums
  S_OUTN = 52,                              // pore cells in the outlet column
  S_GEOM = 56,                              // pore cells, pore-solid faces, sum u_x
  S_IMP = 64,                               // 16: the implicit solver's scalars (host copy)
  S_COUNT = 80                              // slots in d_scal / h_scal
};

// Counter slots in d_counter.
enum { C_RES = 0, C_ULAT = 1, C_CG1 = 2, C_CG2 = 3, C_DT = 4, C_OUT = 5, C_MASS = 6, C_ACC = 7,
       C_GEOM = 8, C_IMP = 9, C_LINK = 10, C_FACE = 11 };

enum { PH_FLOW = 0, PH_CHECK = 1, PH_PSI = 2, PH_NP = 3 };

// Host helpers (api.cu).
cdi_status cdi_fail(cdi_domain *d, cdi_status s, const std::string &msg);
cdi_status cdi_cuda_fail(cdi_domain *d, cudaError_t e, const char *what);
void *cdi_dev_alloc(cdi_domain *d, size_t bytes);
void *cdi_dev_need(cdi_domain *d, size_t bytes);
bool cdi_give_back(cdi_domain *d);
void cdi_timing_begin(cdi_domain *d, cudaEvent_t *a);
void cdi_timing_end(cdi_domain *d, cudaEvent_t a, int phase, int64_t launches);
cudaError_t cdi_timing_resolve(cdi_domain *d);

// Process-wide memory of the autotuners' choices, keyed by the kernel kind,
// lattice, storage precision, species count, problem size and device: a
// second domain of the same size runs the kernels the first one picked (so
// repeated solves time the same code) without re-timing them.
uint64_t cdi_tune_key(int kind, int dim, int prec, int ns, long long n, int extra);
bool cdi_tune_lookup(uint64_t key, int *variant);
void cdi_tune_store(uint64_t key, int variant);

#define CDI_TRY(d, call, what)                           \
  do {                                                   \
    cudaError_t e_ = (call);                             \
    if (e_ != cudaSuccess) return cdi_cuda_fail(d, e_, what); \
  } while (0)

// Kernel-side entry points used by the API layer.
cdi_status cdi_flow_build_flags(cdi_domain *d, void *fflags);
size_t cdi_lists_work_ints(long long n);
cdi_status cdi_flow_build_links(cdi_domain *d, const void *fflags, int *rank_work);
cdi_status cdi_build_lists(cdi_domain *d, const void *fflags, int *work);
cdi_status cdi_flow_run(cdi_domain *d, const cdi_flow_params *p, int64_t *steps,
                        double *res);
cdi_status cdi_flow_export(cdi_domain *d, double U_target);
cdi_status cdi_flow_batch(cdi_domain *const *doms, int n_doms, const cdi_flow_params *p,
                          int64_t *steps, double *res, int *status);
cdi_status cdi_flow_velocity_lattice(cdi_domain *d);
cdi_status cdi_psi_solve(cdi_domain *d, double psi_s, double kdx2, const double *src,
                         double tol, int max_iter, int *iters, double *relres);
cdi_status cdi_psi_coupled(cdi_domain *d);
cdi_status cdi_np_build_flags(cdi_domain *d);
cdi_status cdi_np_build_compact(cdi_domain *d);
cdi_status cdi_np_scatter(cdi_domain *d, int species, double *dst);
cdi_status cdi_np_records_to_planes(cdi_domain *d, int b, float *planes);
cdi_status cdi_np_planes_to_records(cdi_domain *d, const float *planes, int b);
cdi_status cdi_np_faces(cdi_domain *d);
cdi_status cdi_np_init(cdi_domain *d, double dt_s, double *dt_used);
cdi_status cdi_np_dt(cdi_domain *d, double scale, double *dt_out);
cdi_status cdi_np_geometry(cdi_domain *d, double *pores, double *faces, double *sum_ux);
cdi_status cdi_np_sweep(cdi_domain *d, int n, const double *scale, const int *group,
                        void *const *phi_groups, const double *dts, int64_t n_steps,
                        double *gamma, double *cout);
cdi_status cdi_np_batch(cdi_domain *const *doms, int n_doms, int n_combos, const double *scale,
                        const int *group, void *const *phis, const double *dts, int64_t n_steps,
                        double *gamma, double *cout);
cdi_status cdi_flow_scale_to(cdi_domain *d, double scale, void *dst);
void cdi_dev_release(cdi_domain *d, void *p);
cdi_status cdi_np_steps(cdi_domain *d, int64_t n);
cdi_status cdi_np_reduce(cdi_domain *d);
cdi_status cdi_np_column_means(cdi_domain *d, int species);
cdi_status cdi_imp_prepare(cdi_domain *d);
// Nonlinear Poisson-Boltzmann potential (Newton around the device CG).
cdi_status cdi_psi_pb(cdi_domain *d, double psi_s, double kdx2, double tol, int max_iter,
                      int *iters, double *relres);
// Threads per block of LBM / transport launch shape v (0 if v is no shape).
int cdi_lbm_shape_block(int v);
int cdi_np_shape_block(int v);
cdi_status cdi_imp_steps(cdi_domain *d, int64_t n);
