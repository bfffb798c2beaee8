// kernels.cu -- CUDA kernels (sm_103a) for one implicit step of the primitive
// q-NSCH scheme of arXiv:1703.06606: residual with fused norms (Sec. 6.1),
// CH 2x2 Newton Gauss-Seidel and 5x5 Vanka smoothers (Sec. 7.1), FAS
// transfers, frozen-data setup, ghost filling (App. A.6), and FP64 reductions
// for the norms, the mean of p, mass (Thm. 6.1) and energy (Thm. 6.2).
#include <cuda_runtime.h>
#include <math_constants.h>

#include <atomic>
#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "qnsch_dev.cuh"

namespace qn {

constexpr int BX = 32, BY = 8, NT = BX * BY;

// the type a kernel computes in for data of type T: with its contraction fixed
template <typename T, class Form>
using compute_t = Fused<T>;

static inline dim3 grid2(int nx, int ny) { return dim3((nx + BX - 1) / BX, (ny + BY - 1) / BY); }

// number of kernels issued by this library since load (host-side count;
// atomic, since host threads may drive different handles at once)
static std::atomic<long long> g_launches{0};
long long launches_issued() { return g_launches.load(); }

// Programmatic dependent launch (sm_90 and later).  Every kernel of the step is
// launched with programmatic stream serialisation: it is scheduled as the
// blocks of its predecessor in the stream exit, and its threads wait
// (griddepcontrol.wait) until the predecessor grid has completed and its
// memory is visible.  The wait comes before any access to global memory, so
// the order of effects is that of plain stream order; what is saved is part of
// the gap between dependent launches (measured: ~1.3 % of a droplet step).  A
// grid of at most PDL_EARLY blocks also lets its successor's blocks come in
// while it runs (launch_dependents), to fetch their code and parameters and
// wait: 256x512 mixed step 17.9 -> 17.4 ms, 512x512 coupled mixed 7.6 -> 7.4 ms,
// the rest within 1 %.  Not above that: the waiting blocks would take the SMs
// that the running grid's neighbours in time are meant to spread over (every
// grid early: 256x512 FP64 51.6 -> 57.5 ms; up to 76 blocks: a batch of
// instances, whose streams compete for the SMs, 9.8 -> 10.0 ms).
constexpr unsigned PDL_EARLY = 32;
static std::atomic<int> g_pdl{1};
void set_pdl(int on) { g_pdl = on ? 1 : 0; }
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (gridDim.x * gridDim.y * gridDim.z <= PDL_EARLY)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... KArgs, typename... Args>
static void qlaunch(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                    Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g_pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// --------------------------------------------------------------------------
// block reduction helpers (fixed order: deterministic for a fixed launch shape)
// --------------------------------------------------------------------------
// fmax of non-negative values or NaN (which the other operand replaces), by
// their bit patterns: off the FP64 pipe
__device__ __forceinline__ double max_bits(double x, double y) {
  const long long inf = 0x7ff0000000000000LL;
  const long long a = __double_as_longlong(x), b = __double_as_longlong(y);
  return a > inf ? y : b > inf ? x : a > b ? x : y;
}

// sums over a warp of five values each lane holds; lane 0 receives them.  Two
// exchanges first split the values over the lanes (4 + 2 additions), so the
// warp issues 10 FP64 additions instead of 25.
__device__ __forceinline__ void warp_sum5(double& a, double& b, double& c, double& d, double& e) {
  const unsigned FULL = 0xffffffffu;
  const int lane = (threadIdx.y * BX + threadIdx.x) & 31;
  const bool b4 = lane & 16, b3 = lane & 8;
  // lanes 0..15 keep a, b, e, lanes 16..31 keep c, d (and a zero)
  double x = (b4 ? c : a) + __shfl_xor_sync(FULL, b4 ? a : c, 16);
  double y = (b4 ? d : b) + __shfl_xor_sync(FULL, b4 ? b : d, 16);
  double z = e + shfl_xor(e, 16);  // the same on both halves
  // lanes with bit 3 clear keep x, the others y
  double w = (b3 ? y : x) + __shfl_xor_sync(FULL, b3 ? x : y, 8);
  // e on the lanes with bit 2 set in a register of its own: two values, three exchanges
  z += __shfl_xor_sync(FULL, z, 8);
  const bool b2 = lane & 4;
  double wz = (b2 ? z : w) + __shfl_xor_sync(FULL, b2 ? w : z, 4);
  wz += shfl_xor(wz, 2);
  wz += shfl_xor(wz, 1);
  a = __shfl_sync(FULL, wz, 0);
  b = __shfl_sync(FULL, wz, 8);
  c = __shfl_sync(FULL, wz, 16);
  d = __shfl_sync(FULL, wz, 24);
  e = __shfl_sync(FULL, wz, 4);
}

// the rows a thread evaluates: all, or a third of their work (ROLE 0: N_c and
// N_p, which share the flux sum; 1: N_mu; 2: the momentum rows)
constexpr int ROLE_ALL = -1;
template <int ROLE>
__host__ __device__ constexpr bool role_has(int q) {
  return ROLE == ROLE_ALL || (ROLE == 0 ? q == 0 || q == 2 : ROLE == 1 ? q == 1 : q >= 3);
}
// ROLE: only the entries q and 5 + q of the residual families q of that role
template <int NV, int ROLE = -1>
__device__ __forceinline__ void block_sum_store(double (&val)[NV], double* part, int nmax_first) {
  // first `nmax_first` values are reduced with max, the rest with sum.  The
  // max values are non-negative (or NaN), whose bit patterns order as the
  // values do (a NaN above everything), so the warp stage takes their max as
  // 64-bit integers, off the FP64 pipe.
  __shared__ double sh[NT / 32][NV];
  int lane = (threadIdx.y * BX + threadIdx.x) & 31, warp = (threadIdx.y * BX + threadIdx.x) >> 5;
  constexpr bool FIVE = NV == 10 && ROLE == -1;
  if constexpr (FIVE) warp_sum5(val[5], val[6], val[7], val[8], val[9]);
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    if (!role_has<ROLE>(q % 5)) continue;
    double x = val[q];
    if (q < nmax_first) {
      long long b = __double_as_longlong(x);
      for (int o = 16; o > 0; o >>= 1) {
        long long c = __shfl_down_sync(0xffffffffu, b, o);
        b = c > b ? c : b;
      }
      x = __longlong_as_double(b);
    } else if (!FIVE) {
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    }
    if (lane == 0) sh[warp][q] = x;
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      if (!role_has<ROLE>(q % 5)) continue;
      double x = sh[lane & (NT / 32 - 1)][q];  // lane 0 reduces the values of lanes 0 .. NT/32 - 1
      for (int o = NT / 64; o > 0; o >>= 1) {
        const double y = __shfl_down_sync(0xffffffffu, x, o);
        x = q < nmax_first ? max_bits(x, y) : x + y;
      }
      if (lane == 0) part[(blockIdx.y * gridDim.x + blockIdx.x) * NV + q] = x;
    }
  }
}

// Sum (or max) nparts rows of nv <= 32 partials in a fixed order, in one block:
// consecutive threads read consecutive partials (a thread's all of one
// column), and a warp then adds each column's share.  One block's dependent
// loads bound it: with 1024 threads reading in rows 11.6 -> 6 us on 256x512 and
// 41.7 -> 12 us on 1024x4096 (256 threads, a column each, before).
constexpr int FIN_NT = 1024;
__global__ void __launch_bounds__(FIN_NT) k_finalize(const double* part, int nparts, int nv,
                                                     int nmax_first, double scale_sum, double* out) {
  pdl_enter();
  __shared__ double sh[FIN_NT];
  const int stride = FIN_NT / nv * nv, q = threadIdx.x % nv;
  const bool mx = q < nmax_first;
  double acc = 0.0;
  if ((int)threadIdx.x < stride) {
    const long long n = (long long)nparts * nv;
#pragma unroll 4
    for (long long p = threadIdx.x; p < n; p += stride) {
      const double x = part[p];
      if (mx) acc = max_bits(acc, x);
      else acc += x;
    }
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w >= nv) return;
  const bool wmx = w < nmax_first;
  double x = 0.0;
  for (int p = w + lane * nv; p < stride; p += 32 * nv) {
    if (wmx) x = max_bits(x, sh[p]);
    else x += sh[p];
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double y = __shfl_down_sync(0xffffffffu, x, o);
    x = wmx ? max_bits(x, y) : x + y;
  }
  if (lane == 0) out[w] = wmx ? x : x * scale_sum;
}

// --------------------------------------------------------------------------
// residual r = f - N(x) (mode 0, optional norms) or f += N(x) (mode 1)
// thread (i,j): cell families at (i,j), u-edge (i,j) and v-edge (i,j)
// --------------------------------------------------------------------------
// The FP64 primitive operator in the fewest FP64 instructions (the pipe that
// bounds the kernels that evaluate it): sums over the four faces of unscaled
// differences, scaled once by the level's constants.
// sum over the faces of (m(c^n) of both cells) (d mu + alpha d p): 2 h^2 Pe
// times the diffusion of N_c.  Differences of mu and of p first: those of
// mu + alpha p would round at alpha p's own size, 20 to 300 times the error on
// 64 to 1024 cells across, and grow as 1/h^2 in the row.
template <typename T, class LV>
__device__ __forceinline__ T flux_sum(const Prm<T>& P, const LV& L, int k) {
  const int W = L.pitch;
  auto mob = L.mobn; auto mu = L.mu; auto p = L.p;
  const int off[4] = {1, -1, W, -W};
  T mk = mob[k], s = T(0), sp = T(0);
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    int q = k + off[f];
    T m = mk + mob[q], dmu = mu[q] - mu[k], dp = p[q] - p[k];
    if constexpr (sizeof(T) == 8) {  // the two fields' sums apart: alpha once, one rounding a face less
      s += m * dmu;
      sp += m * dp;
    } else {
      s += m * (dmu + P.alpha * dp);
    }
  }
  if constexpr (sizeof(T) == 8) s += P.alpha * sp;
  return s;
}
// the advection (e1e2) of N_c
template <class LV>
__device__ __forceinline__ typename LV::real adv_sum(const LV& L, int k) {
  typedef typename LV::real T;
  const int W = L.pitch;
  auto rn = L.rhon;
  return rn[k + 1] * L.Tx[k] * L.u[k] + rn[k - 1] * L.Tx[k - 1] * L.u[k - 1] +
         rn[k + W] * L.Ty[k] * L.v[k] + rn[k - W] * L.Ty[k - W] * L.v[k - W];
}
// (pm-num-chem) with its constants folded: with S = rho + rho^n, A(c) =
// c (c - 1), 8 rho^{n+1/2} g = S (A + A^n)(c + c^n - 1) and 8 (F + F^n)/2 =
// A^2 + (A^n)^2
template <typename T, class LV>
__device__ __forceinline__ T chem_full(const Prm<T>& P, const LV& L, int k, T rk,
                                       const T (&rq)[4]) {
  const int W = L.pitch;
  auto c = L.c; auto cn = L.cn; auto rn = L.rhon;
  const int off[4] = {1, -1, W, -W};
  T ck = c[k], cnk = cn[k], rnk = rn[k];
  T S = rk + rnk, ch = ck + cnk;
  T A = ck * ck - ck, An = cnk * cnk - cnk;
  T G2 = T(0), div = T(0), SD = T(0);
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    int q = k + off[f];
    T d = c[q] - ck, D = (c[q] + cn[q]) - ch;
    G2 += d * d;
    div += (rq[f] + rn[q]) * D;
    SD += D;
  }
  div += S * SD;
  T E = L.k.K8 * (A * A + An * An) + L.k.L4 * (L.k.hih2 * G2 + L.Gn[k]);
  return rk * L.mu[k] + L.k.L8 * div - L.k.K8 * (S * ((A + An) * (ch - T(1)))) +
         P.alpha * rk * rnk * E;
}

// the residual's five rows at one cell: r = f - N(x) (MODE 0) or f + N(x) (MODE 1)
template <typename T>
struct Rows5 {
  T r[5];
};
// at thread (i,j): cell families at (i,j), u-edge (i,j) and v-edge (i,j); the
// edge rows also on boundary edges (padded arrays), which are masked later
template <typename T, int MODE, class Form, int ROLE, class LV>
__device__ __forceinline__ Rows5<T> residual_rows5(const Prm<T>& P, const LV& L, int i, int j) {
  const int k = L.at(i, j), W = L.pitch;
  constexpr bool CP = role_has<ROLE>(0), MU = role_has<ROLE>(1), UV = role_has<ROLE>(3);
  const T f[5] = {CP ? L.fc[k] : T(0), MU ? L.fmu[k] : T(0), CP ? L.fp[k] : T(0),
                  UV ? L.fu[k] : T(0), UV ? L.fv[k] : T(0)};
  T n[5] = {T(0), T(0), T(0), T(0), T(0)};
  if constexpr (std::is_same<Form, ErrForm>::value) {
    const ErrCell<T> X = err_cell(P, L, k);
    T flux = flux_sum(P, L, k);
    n[0] = err_c(P, L, k, X.r[0]) - L.k.dif * flux;
    n[1] = err_mu(P, L, k, X);
    n[2] = (L.u[k] - L.u[k - 1] + L.v[k] - L.v[k - W]) * L.ih - L.k.adif * flux;
    n[3] = err_row(P, L, 0, k, X.r[0] + X.r[1], X.dr[0] + X.dr[1]);
    n[4] = err_row(P, L, 1, k, X.r[0] + X.r[3], X.dr[0] + X.dr[3]);
  } else {
    constexpr bool PROJ = std::is_same<Form, ProjForm>::value;
    // rho(c) of the cell and its neighbours, shared by the rows
    auto rc = L.rhoc;
    const T rk = rc[k];
    const T rq[4] = {rc[k + 1], rc[k - 1], rc[k + W], rc[k - W]};
    if constexpr (CP) {
      T flux = flux_sum(P, L, k);
      if constexpr (PROJ) {
        T w[4];
        proj_faces(P, L, i, j, rk, rq, w);
        n[0] = opp_c_w(P, L, k, rq, w, flux);
        n[2] = opp_p_w(L, w, flux);
      } else {
        n[0] = rk * (L.c[k] - L.cn[k]) * P.idt + adv_sum(L, k) - L.k.dif * flux;
        n[2] = (L.u[k] - L.u[k - 1] + L.v[k] - L.v[k - W]) * L.ih - L.k.adif * flux;
      }
    }
    if constexpr (MU) {
      n[1] = chem_full(P, L, k, rk, rq);
      if constexpr (PROJ) n[1] += (L.rhon[k] - rk) * L.mu[k];  // rho^n in front of mu
    }
    if constexpr (UV) {
      n[3] = full_mom_row<PROJ>(L, 0, k, rk + rq[0]);
      n[4] = full_mom_row<PROJ>(L, 1, k, rk + rq[2]);
    }
  }
  Rows5<T> X;
#pragma unroll
  for (int q = 0; q < 5; ++q) X.r[q] = MODE == 0 ? f[q] - n[q] : f[q] + n[q];
  return X;
}
// stores them (MODE 0: into r, MODE 1: into f) and adds to val: the largest |r|
// and the sum of r^2 per family (MODE 0 with norms: a cycle's own residuals need
// none, and in FP32 their conversions and sums, ten FP64 instructions a cell,
// were a quarter of the launch: 219 -> 164 us on 1024x4096)
template <typename T, int MODE, int ROLE, class LV>
__device__ __forceinline__ void residual_store(const LV& L, int i, int j, const Rows5<T>& X,
                                               double (&val)[10], bool norms) {
  const int k = L.at(i, j);
  const bool own[5] = {true, true, true, i <= L.uhi(), j < L.m2};
  const bool has[5] = {role_has<ROLE>(0), role_has<ROLE>(1), role_has<ROLE>(2),
                       role_has<ROLE>(3) && own[3], role_has<ROLE>(4) && own[4]};
  if (has[0]) (MODE == 0 ? L.rc[k] : L.fc[k]) = X.r[0];
  if (has[1]) (MODE == 0 ? L.rmu[k] : L.fmu[k]) = X.r[1];
  if (has[2]) (MODE == 0 ? L.rp[k] : L.fp[k]) = X.r[2];
  if (has[3]) (MODE == 0 ? L.ru[k] : L.fu[k]) = X.r[3];
  if (has[4]) (MODE == 0 ? L.rv[k] : L.fv[k]) = X.r[4];
  if (MODE == 0 && norms) {
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      if (!role_has<ROLE>(q)) continue;
      const double a = own[q] ? (double)X.r[q] : 0.0;
      // |r| >= 0 or NaN: the bit patterns order as the values
      const long long b = __double_as_longlong(fabs(a)), m = __double_as_longlong(val[q]);
      val[q] = __longlong_as_double(b > m ? b : m);
      val[5 + q] += a * a;
    }
  }
}
template <typename T, int MODE, class Form, class LV>
__device__ __forceinline__ void residual_cell(const Prm<T>& P, const LV& L, int i, int j,
                                              double (&val)[10], bool norms) {
  residual_store<T, MODE, ROLE_ALL>(L, i, j, residual_rows5<T, MODE, Form, ROLE_ALL>(P, L, i, j), val,
                                    norms);
}

// ROWS > 1 (large levels): each thread takes ROWS / 2 pairs of rows BY apart, so
// that the norms' reduction is shared by ROWS cells.  Both rows of a pair are
// evaluated before either is stored: the second's loads would wait behind
// stores they might alias.
template <typename T, int MODE, class Form, int ROWS>
__global__ void __launch_bounds__(NT, 2) k_residual(Prm<T> P, Lv<T> L, double* part) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x + 1;
  int j = blockIdx.y * (ROWS * BY) + threadIdx.y + 1;
  const bool norms = MODE == 0 && part;
  double val[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};  // max x5 then sum of squares x5
  if (ROWS == 1) {
    if (i <= L.m1 && j <= L.m2) residual_cell<T, MODE, Form>(P, L, i, j, val, norms);
  } else {
#pragma unroll 1
    for (int r = 0; r < ROWS; r += 2, j += 2 * BY) {
      if (i > L.m1 || j > L.m2) break;
      const bool two = j + BY <= L.m2;
      const Rows5<T> A = residual_rows5<T, MODE, Form, ROLE_ALL>(P, L, i, j);
      const Rows5<T> B = residual_rows5<T, MODE, Form, ROLE_ALL>(P, L, i, two ? j + BY : j);
      residual_store<T, MODE, ROLE_ALL>(L, i, j, A, val, norms);
      if (two) residual_store<T, MODE, ROLE_ALL>(L, i, j + BY, B, val, norms);
    }
  }
  if (norms) block_sum_store<10>(val, part, 5);
}

// The rows of a cell by three threads (ROLE: the block's z), for levels that
// leave most of the FP64 pipes idle: a thread's chain of FP64 instructions, 64
// cycles each, is what such a launch takes, and the longest third is 50 of the
// 137.  A role's blocks write its families' entries of the partials.
template <typename T, int MODE, class Form, int ROLE>
__device__ __forceinline__ void residual_role(const Prm<T>& P, const Lv<T>& L, double* part) {
  int i = blockIdx.x * BX + threadIdx.x + 1;
  int j = blockIdx.y * BY + threadIdx.y + 1;
  const bool norms = MODE == 0 && part;
  double val[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  if (i <= L.m1 && j <= L.m2)
    residual_store<T, MODE, ROLE>(L, i, j, residual_rows5<T, MODE, Form, ROLE>(P, L, i, j), val, norms);
  if (norms) block_sum_store<10, ROLE>(val, part, 5);
}
template <typename T, int MODE, class Form>
__global__ void __launch_bounds__(NT, 2) k_residual_split(Prm<T> P, Lv<T> L, double* part) {
  pdl_enter();
  if (blockIdx.z == 0) residual_role<T, MODE, Form, 0>(P, L, part);
  else if (blockIdx.z == 1) residual_role<T, MODE, Form, 1>(P, L, part);
  else residual_role<T, MODE, Form, 2>(P, L, part);
}

// rows per residual thread on level L: two on levels of at least 65536 cells,
// eight where that still leaves the GPU several blocks an SM (2^21 cells: 1024
// blocks), so that one block sums a quarter of the partials (with the wider
// k_finalize 30 us of a 1024x4096 residual and its norms)
template <typename T>
static int residual_rows(const Lv<T>& L) {
  const long long n = (long long)L.m1 * L.m2;
  return n >= (1LL << 21) ? 8 : n >= 65536 ? 2 : 1;
}

// --------------------------------------------------------------------------
// CH step 1 of Sec. 7.1: Newton step on the 2x2 system (N_c, N_mu) in (c, mu)
// of each cell with (i + j) % 2 == colour; neighbours frozen.  Faces on
// Neumann walls do not contribute (their ghost follows the cell).
// --------------------------------------------------------------------------
// ch_system for the full iterate (PROJ: the projection method's form), with the
// constants and the terms
// common to the residuals and the Jacobian folded (chem_full's notation; E =
// K ((F + F^n)/2) + (Lam/4) Gbar): about 119 FP64 instructions where the
// unfolded sums take about 190.  On a wall face the ghost's c and c^n are the
// cell's own, so its differences vanish and only the coefficients of c (2 rho
// sums) and the mobilities need the face left out.
template <bool PROJ, typename T, class LV>
__device__ __forceinline__ void ch_system_full(const Prm<T>& P, const LV& L, int i, int j,
                                               T (&J)[2][2], T (&R)[2]) {
  const int W = L.pitch;
  const int k = L.at(i, j);
  const int off[4] = {1, -1, W, -W};
  const bool wall[4] = {!L.px && i == L.m1, !L.px && i == 1, j == L.m2, j == 1};
  auto c = L.c; auto cn = L.cn; auto rn = L.rhon; auto rc = L.rhoc; auto mob = L.mobn; auto mu = L.mu; auto p = L.p;
  T ck = c[k], cnk = cn[k], rk = rc[k], rnk = rn[k], muk = mu[k];
  T mk = mob[k], pk = p[k];
  T S = rk + rnk, ch = ck + cnk;
  T flux = T(0), fluxp = T(0), sm = T(0), G2 = T(0), sd = T(0), div = T(0), SD = T(0), SW = T(0);
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    const int q = k + off[f];
    T m = mk + mob[q], cq = c[q];
    flux += m * (mu[q] - muk);  // flux_sum's two sums
    fluxp += m * (p[q] - pk);
    T d = cq - ck, D = (cq + cn[q]) - ch, H = rc[q] + rn[q];
    G2 += d * d;
    sd += d;
    div += H * D;
    SD += D;
    sm += wall[f] ? T(0) : m;
    SW += wall[f] ? T(0) : H;
  }
  const int open = 4 - (wall[0] + wall[1] + wall[2] + wall[3]);
  SW += (open == 4 ? T(4) : open == 3 ? T(3) : open == 2 ? T(2) : open == 1 ? T(1) : T(0)) * S;
  div += S * SD;
  flux += P.alpha * fluxp;
  T dck = ck - cnk, ar = -P.alpha * rk, drho = ar * rk, r = ar * rnk;
  T dr = -P.alpha * rnk * drho;
  T A = ck * ck - ck, An = cnk * cnk - cnk, sA = A + An, t = ch - T(1), g4 = sA * t;
  T Gs = L.k.hih2 * G2 + L.Gn[k];
  T E = L.k.K8 * (A * A + An * An) + L.k.L4 * Gs;
  R[1] = (PROJ ? rnk : rk) * muk - L.fmu[k] + L.k.L8 * div - L.k.K8 * (S * g4) - r * E;
  T tc = T(2) * ck - T(1);
  J[0][1] = L.k.dif * sm;
  J[1][0] = drho * ((PROJ ? T(0) : muk) + L.k.L8 * SD - L.k.K8 * g4) - L.k.K8 * (S * (tc * t + sA)) -
            r * (L.k.K4 * (A * tc) - L.k.L4h * sd) - dr * E - L.k.L8 * SW;
  if constexpr (PROJ) {
    // projection method: rho^n in the time derivative and in front of mu; the
    // advection a(rho(c) D c u^{n+1}) differentiated in c_ij through D c only,
    // with rho(c) of the neighbours and u^{n+1} at the iterate (the smoother's
    // choice; the fixed point is the scheme's)
    const T rq[4] = {rc[k + 1], rc[k - 1], rc[k + W], rc[k - W]};
    T w[4];  // the face velocities u^{n+1} (E, W, N, S)
    proj_faces(P, L, i, j, rk, rq, w);
    R[0] = opp_c_w(P, L, k, rq, w, flux) - L.fc[k];
    J[0][0] = rnk * P.idt + L.k.hih * (rq[1] * w[1] - rq[0] * w[0] + rq[3] * w[3] - rq[2] * w[2]);
    J[1][1] = rnk;
  } else {
    R[0] = rk * dck * P.idt - L.fc[k] + adv_sum(L, k) - L.k.dif * flux;
    J[0][0] = (rk + drho * dck) * P.idt;
    J[1][1] = rk;
  }
}

// ch_system for the error equation: the residuals of err_c and err_mu, and
// ch_system_full's Jacobian at the full values C + e, Mu + e_mu
template <typename T, class LV>
__device__ __forceinline__ void ch_system_err(const Prm<T>& P, const LV& L, int i, int j,
                                              const ErrCell<T>& X, T (&J)[2][2], T (&R)[2]) {
  const int W = L.pitch;
  const int k = L.at(i, j);
  const int off[5] = {0, 1, -1, W, -W};
  const bool wall[5] = {false, !L.px && i == L.m1, !L.px && i == 1, j == L.m2, j == 1};
  auto mob = L.mobn;
  R[0] = err_c(P, L, k, X.r[0]) - L.k.dif * flux_sum(P, L, k) - L.fc[k];
  R[1] = err_mu(P, L, k, X) - L.fmu[k];
  T ck = X.B[0] + X.e[0], cnk = L.cn[k], rk = X.r[0], rnk = X.rn[0], mk = mob[k];
  T muk = L.Bmu[k] + L.mu[k];
  T S = rk + rnk, ch = ck + cnk;
  T sm = T(0), G2 = T(0), sd = T(0), SD = T(0), SW = T(0);
#pragma unroll
  for (int f = 1; f < 5; ++f) {
    T cq = X.B[f] + X.e[f], d = cq - ck;
    G2 += d * d;
    sd += d;
    SD += (cq + L.cn[k + off[f]]) - ch;
    sm += wall[f] ? T(0) : mk + mob[k + off[f]];
    SW += wall[f] ? T(0) : S + (X.r[f] + X.rn[f]);
  }
  T dck = ck - cnk, ar = -P.alpha * rk, drho = ar * rk, r = ar * rnk;
  T dr = -P.alpha * rnk * drho;
  T A = ck * ck - ck, An = cnk * cnk - cnk, sA = A + An, t = ch - T(1), g4 = sA * t;
  T Gs = L.k.hih2 * G2 + L.Gn[k];
  T E = L.k.K8 * (A * A + An * An) + L.k.L4 * Gs;
  T tc = T(2) * ck - T(1);
  J[0][0] = (rk + drho * dck) * P.idt;
  J[0][1] = L.k.dif * sm;
  J[1][0] = drho * (muk + L.k.L8 * SD - L.k.K8 * g4) - L.k.K8 * (S * (tc * t + sA)) -
            r * (L.k.K4 * (A * tc) - L.k.L4h * sd) - dr * E - L.k.L8 * SW;
  J[1][1] = rk;
}

// The 2x2 CH system of cell (i,j): residuals R = N - f of (N_c, N_mu) and their
// Jacobian J in (c, mu), neighbours frozen, at the full values c, mu
template <typename T, class Form, class LV>
__device__ __forceinline__ void ch_system(const Prm<T>& P, const LV& L, int i, int j,
                                          T (&J)[2][2], T (&R)[2]) {
  if constexpr (std::is_same<Form, ErrForm>::value)
    ch_system_err(P, L, i, j, err_cell(P, L, L.at(i, j)), J, R);
  else
    ch_system_full<std::is_same<Form, ProjForm>::value>(P, L, i, j, J, R);
}

template <typename T, class Form, class LV>
__device__ __forceinline__ void ch_cell(const Prm<T>& P, const LV& L, int i, int j) {
  T J[2][2], R[2];
  ch_system<T, Form>(P, L, i, j, J, R);
  T idet = qrcp(J[0][0] * J[1][1] - J[0][1] * J[1][0]);
  T dc = (J[1][1] * R[0] - J[0][1] * R[1]) * idet;
  T dm = (J[0][0] * R[1] - J[1][0] * R[0]) * idet;
  int k = L.at(i, j);
  const bool ghosts = has_ghosts(L, i, j);
  const T cnew = L.c[k] - dc, mnew = L.mu[k] - dm;
  put_cell(L, L.c, i, j, ghosts, cnew);
  if constexpr (!std::is_same<Form, ErrForm>::value)
    put_cell(L, L.rhoc, i, j, ghosts, rho_of(P, cnew));
  put_cell(L, L.mu, i, j, ghosts, mnew);
}

// Vanka colour of cell (i,j): (2i + j) mod 8 (c8: periodic x, m1 = 0 mod 4) or
// (i + 2j) mod kcol (kcol = 5 with walls, the smallest divisor >= 5 of m1 otherwise).
// First cell i0 >= 1 of colour `colour` in row j and the stride between cells
// of that colour in the row; false if the row has none
template <class LV>
__device__ __forceinline__ bool colour_row(const LV& L, int colour, int j, int& i0, int& stride) {
  if (L.c8) {
    int d = (colour - j) & 7;
    if (d & 1) return false;
    i0 = d >> 1;
    if (i0 == 0) i0 = 4;
    stride = 4;
  } else {
    const int K = L.kcol;
    int y = colour + 2 * (K - (j - K * L.kdiv.div(j)));  // (colour - 2j) mod K, plus at most 2K
    y = y >= 2 * K ? y - 2 * K : y;
    y = y >= K ? y - K : y;
    i0 = y == 0 ? K : y;
    stride = K;
  }
  return true;
}

// slots of Vanka colour `col`: slot t -> row j0 + rstep * (t / mpr), t % mpr-th
// cell of that row's colour
struct ColourSlots {
  int j0, rstep, mpr, n;
};

template <class LV>
__host__ __device__ __forceinline__ ColourSlots vanka_slots(const LV& L, int col) {
  ColourSlots cs;
  cs.j0 = L.c8 && ((col - 1) & 1) ? 2 : 1;  // eight colours: rows with (col - j) even
  cs.rstep = L.c8 ? 2 : 1;
  cs.mpr = L.vrow.d;
  cs.n = cs.j0 > L.m2 ? 0 : (((L.m2 - cs.j0) >> (cs.rstep - 1)) + 1) * cs.mpr;
  return cs;
}

template <class LV>
__device__ __forceinline__ bool vanka_slot_cell(const LV& L, int col, const ColourSlots& cs, int t,
                                                int& i, int& j) {
  const int r = L.vrow.div(t);
  j = cs.j0 + cs.rstep * r;
  int i0, stride;
  if (!colour_row(L, col, j, i0, stride)) return false;
  i = i0 + stride * (t - r * cs.mpr);
  return i <= L.m1;
}

// cell of slot t of CH colour `colour` ((i + j) % 2, rows packed); false past the row's end
template <class LV>
__device__ __forceinline__ bool ch_slot_cell(const LV& L, int colour, int t, int& i, int& j) {
  const int r = L.crow.div(t);
  j = r + 1;
  i = (((colour - j) & 1) ? 1 : 2) + 2 * (t - r * L.crow.d);
  return i <= L.m1;
}

// cells of CH colour `colour` ((i + j) % 2), packed: slot t -> row t / mpr + 1
template <typename T, class Form>
__global__ void __launch_bounds__(64, 4) k_ch(Prm<T> P, Lv<T> L, int colour) {
  pdl_enter();
  int t = blockIdx.x * 64 + threadIdx.x, i, j;
  if (t >= L.crow.d * L.m2 || !ch_slot_cell(L, colour, t, i, j)) return;
  ch_cell<T, Form>(P, L, i, j);
}

// sum over the four lanes of a team (lanes 4t .. 4t+3)
template <typename T>
__device__ __forceinline__ T team_sum(T v) {
  v += shfl_xor(v, 1);
  return v + shfl_xor(v, 2);
}

// u^{n+1} at face q (W, E, S, N) of cell k (0 on a wall face), as proj_faces
// gives it: rho(c) of the cell rk and of the face's neighbour rn
template <typename T, class LV>
__device__ __forceinline__ T proj_face_team(const Prm<T>& P, const LV& L, int k, int q, bool open, T rk,
                                            T rn) {
  const int d = q >> 1, off = d ? L.pitch : 1;
  const bool hi = q & 1;  // E or N: the face's velocity sits at k
  const int a = hi ? k : k - off;
  auto vel = L.pair(d, L.u, L.v);
  auto c = L.c;
  auto mu = L.mu;
  auto p = L.p;
  T ra = hi ? rk : rn, rb = hi ? rn : rk;
  return open ? vel[a] + proj_kick(L, ra, rb, mu[a], mu[a + off], c[a + off] - c[a], p[a + off] - p[a]) -
                    (d ? L.k.gdt : T(0))
              : T(0);
}

// rho(c) of the full value at cell k and, on error levels, its difference to
// the base's: what the rows of a team's lane need of a cell
template <typename T>
struct RhoPair {
  T r, d;
};
template <typename T, class Form, class LV>
__device__ __forceinline__ RhoPair<T> rho_pair(const Prm<T>& P, const LV& L, int k) {
  const T r = Form::rho(P, L, k);
  if constexpr (std::is_same<Form, ErrForm>::value) return {r, rsec_(P, r, L.rB[k]) * L.c[k]};
  else return {r, T(0)};
}

// Whether small launches in T give a visit four lanes.  In FP64 a warp's
// instruction holds its pipe for 64 cycles or more whatever its lanes do, so a
// visit split over four lanes is a shorter chain.  In FP32 the chain is loads
// and their latency, and one lane that has all of them in flight at once
// (launch bounds that leave it the registers) is as fast on the smallest level
// and twice as fast on the largest: coupled visits 4.4 us a colour on 14x14 to
// 56x56 levels and 6.1 us on 448x448 with one lane, 4.5 and 12.5 us (512x512)
// with four.
template <typename T>
constexpr bool lane_teams = sizeof(T) == 8;

// sums over the four lanes of a team of eight values each lane holds, every
// lane receiving all eight: the first exchange halves what a lane adds up
// (4 + 2 additions a lane where eight butterflies take 16; each addition is
// that of team_sum, so the sums are the same)
template <typename T>
__device__ __forceinline__ void team_sum8(T (&v)[8]) {
  const int lane = threadIdx.x & 31;
  const bool b0 = lane & 1, b1 = lane & 2;
  T r[4], t[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    T send = b0 ? v[i] : v[i + 4], keep = b0 ? v[i + 4] : v[i];
    r[i] = keep + shfl_xor(send, 1);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    T send = b1 ? r[i] : r[i + 2], keep = b1 ? r[i + 2] : r[i];
    t[i] = keep + shfl_xor(send, 2);
  }
#pragma unroll
  for (int m = 0; m < 8; ++m)
    v[m] = shfl_from(t[m & 1], (lane & 28) | (m >> 2) | (m & 2));
}

// The CH rows of cell (i,j) for a team of four lanes (lane & 3 = q: face W,
// E, S, N; open = face q is not a wall): residuals Rc = N_c - f_c,
// Rm = N_mu - f_mu and the 2x2 Jacobian of ch_system, and for the coupled
// block the open-face sum of A m, the diffusion flux sum, d rho/dc and face
// q's rho^n D c^n / 2.  Lane q evaluates face q's terms of N_c, N_mu (err_c
// and err_mu on error levels) and of the Jacobian's face
// sums; butterflies add them and every lane forms the cell terms.
template <typename T>
struct ChRows {
  T Rc, Rm, J11, J12, J21, J22;
  T sm, sflux, drho, gq;
};

// ch_team_rows for the full iterate: ch_system_full's sums, a face a lane
template <bool PROJ, typename T, class LV>
__device__ __forceinline__ ChRows<T> ch_team_rows_full(const Prm<T>& P, const LV& L, int i, int j,
                                                       int q, bool open, T rk, T rq) {
  const int W = L.pitch;
  const int d = q >> 1;
  const int k = L.at(i, j);
  const int nq = k + (q == 0 ? -1 : q == 1 ? 1 : q == 2 ? -W : W);
  const int kf = q == 0 ? k - 1 : (q == 2 ? k - W : k);  // edge of face q
  auto c = L.c; auto cn = L.cn; auto rn = L.rhon; auto mob = L.mobn;
  T ck = c[k], cnk = cn[k], rnk = rn[k], muk = L.mu[k];
  T cq = c[nq], rnq = rn[nq];
  T gq = rnq * L.pair(d, L.Tx, L.Ty)[kf];  // rho^n D c^n / 2 at face q
  T m = mob[k] + mob[nq];
  T S = rk + rnk, ch = ck + cnk, dq = cq - ck, D = (cq + cn[nq]) - ch, H = rq + rnq;
  // the projection method advects rho(c) c with u^{n+1} at the face
  T wq = T(0), rw = T(0);
  if constexpr (PROJ) {
    wq = proj_face_team(P, L, k, q, open, rk, rq);
    rw = rq * wq;
  }
  T v[8] = {m * ((L.mu[nq] - muk) + P.alpha * (L.p[nq] - L.p[k])),  // differences first (flux_sum)
            open ? m : T(0),
            PROJ ? rw * ((q & 1) ? dq : -dq) : gq * L.pair(d, L.u, L.v)[kf],
            dq * dq,
            dq,
            (H + S) * D,
            D,
            open ? H + S : T(0)};
  team_sum8(v);
  const T flux = v[0], sm = v[1], adv = v[2], G2 = v[3], sd = v[4], div = v[5], SD = v[6],
          SW = v[7];
  T dck = ck - cnk, ar = -P.alpha * rk, drho = ar * rk, r = ar * rnk;
  T dr = -P.alpha * rnk * drho;
  T A = ck * ck - ck, An = cnk * cnk - cnk, sA = A + An, t = ch - T(1), g4 = sA * t;
  T Gs = L.k.hih2 * G2 + L.Gn[k];
  T E = L.k.K8 * (A * A + An * An) + L.k.L4 * Gs;
  T tc = T(2) * ck - T(1);
  ChRows<T> R;
  if constexpr (PROJ) {
    R.Rc = rnk * dck * P.idt - L.fc[k] + L.k.hih * adv - L.k.dif * flux;
    R.J11 = rnk * P.idt + L.k.hih * team_sum<T>((q & 1) ? -rw : rw);
    R.J22 = rnk;
  } else {
    R.Rc = rk * dck * P.idt - L.fc[k] + adv - L.k.dif * flux;
    R.J11 = (rk + drho * dck) * P.idt;
    R.J22 = rk;
  }
  R.Rm = (PROJ ? rnk : rk) * muk - L.fmu[k] + L.k.L8 * div - L.k.K8 * (S * g4) - r * E;
  R.J12 = L.k.dif * sm;
  R.J21 = drho * ((PROJ ? T(0) : muk) + L.k.L8 * SD - L.k.K8 * g4) - L.k.K8 * (S * (tc * t + sA)) -
          r * (L.k.K4 * (A * tc) - L.k.L4h * sd) - dr * E - L.k.L8 * SW;
  R.sm = sm;
  R.sflux = flux;
  R.drho = drho;
  R.gq = gq;
  return R;
}

template <typename T, class Form, class LV>
__device__ __forceinline__ ChRows<T> ch_team_rows(const Prm<T>& P, const LV& L, int i, int j, int q,
                                                  bool open, RhoPair<T> ra, RhoPair<T> rb) {
  if constexpr (!std::is_same<Form, ErrForm>::value) {
    return ch_team_rows_full<std::is_same<Form, ProjForm>::value>(P, L, i, j, q, open, ra.r, rb.r);
  } else {
    const int W = L.pitch;
    const int d = q >> 1;
    const T ih2 = L.ih2;
    int k = L.at(i, j);
    auto mob = L.mobn; auto cn = L.cn; auto rn = L.rhon;
    const int nq = k + (q == 0 ? -1 : q == 1 ? 1 : q == 2 ? -W : W);
    const int kf = q == 0 ? k - 1 : (q == 2 ? k - W : k);  // edge of face q
    // full values at the cell and at the face's neighbour
    T ck = Form::val_c(L, k), cnk = cn[k], mk = Form::val_mu(L, k), rnk = rn[k];
    T rho = ra.r;
    T cq = Form::val_c(L, nq), rq = rb.r;
    T drho = -P.alpha * rho * rho;
    T rh = T(0.5) * (rho + rnk);
    T chk = ck + cnk;
    T am = mob[nq] + mob[k];
    T gq = rn[nq] * L.pair(d, L.Tx, L.Ty)[kf];  // rho^n D c^n / 2 at face q
    T dlt = cq - ck;
    // face sums: diffusion flux (N_c and the mass row), sum A m over open faces,
    // advection of N_c, and the Jacobian's G, dG/dc and d(div)/dc terms
    T sflux = team_sum<T>(am * ((L.mu[nq] - L.mu[k]) + P.alpha * (L.p[nq] - L.p[k])));
    T sm = team_sum<T>(open ? am : T(0));
    T sadv = team_sum<T>(gq * L.pair(d, L.u, L.v)[kf]);
    T G2 = team_sum<T>(dlt * dlt);
    T dG = team_sum<T>(open ? -dlt : T(0));
    T dd = team_sum<T>(open ? T(0.5) * drho * ((cq + cn[nq]) - chk) - (rh + T(0.5) * (rq + rn[nq])) : T(0));
    auto e = L.c; auto B = L.Bc;
    T ek = e[k], Ck = B[k];
    T Nc = ek * (rho + rsec_(P, rho, L.rB[k]) * L.Bdc[k]) * P.idt + sadv - L.k.dif * sflux;
    T dC = B[nq] - Ck, de = e[nq] - ek;
    T dr = ra.d;
    T drq = rb.d;
    T chP = Ck + cnk;
    T sdGe = team_sum<T>(de * (T(2) * dC + de));
    T sGC = team_sum<T>(dC * dC);
    T sddiv = team_sum<T>((rh + T(0.5) * (rq + rn[nq])) * de + T(0.5) * (dr + drq) * ((B[nq] + cn[nq]) - chP));
    T r_new = rsec_(P, rho, rnk);
    T d_r = -P.alpha * rnk * dr;
    T dF = gsec(ck, Ck) * ek;
    T dbulk = rh * dgsec(Ck, cnk, ek) + T(0.5) * dr * gsec(Ck, cnk) + T(0.5) * dF * r_new +
              T(0.5) * (Fdw(Ck) + Fdw(cnk)) * d_r;
    T dgrad = T(0.25) * P.Lam * (T(0.5) * sdGe * ih2 * r_new + (T(0.5) * sGC * ih2 + L.Gn[k]) * d_r);
    T Nm = rho * L.mu[k] + dr * L.Bmu[k] - P.K * dbulk - dgrad + P.Lam * T(0.25) * ih2 * sddiv;
    ChRows<T> R;
    R.Rc = Nc - L.fc[k];
    R.Rm = Nm - L.fmu[k];
    T r = -P.alpha * rho * rnk, drr = -P.alpha * drho * rnk;
    R.J11 = (rho + drho * (ck - cnk)) * P.idt;
    R.J12 = L.k.dif * sm;
    T Gs = T(0.5) * G2 * ih2 + L.Gn[k];
    T dbulkJ = T(0.5) * drho * gsec(ck, cnk) + rh * gsec_da(ck, cnk) + T(0.5) * fdw(ck) * r +
               T(0.5) * (Fdw(ck) + Fdw(cnk)) * drr;
    T dgradJ = T(0.25) * P.Lam * (dG * ih2 * r + Gs * drr);
    R.J21 = drho * mk - P.K * dbulkJ - dgradJ + P.Lam * T(0.25) * ih2 * dd;
    R.J22 = rho;
    R.sm = sm;
    R.sflux = sflux;
    R.drho = drho;
    R.gq = gq;
    return R;
  }
}

// CH step of cell (i,j) by a team of four lanes (ch_team_rows), every lane
// solving the 2x2 Newton step; lane 0 stores.  All 32 lanes of the warp call
// this (ok = false: a spare team on cell (1,1), no store).
template <typename T, class Form, class LV>
__device__ __forceinline__ void ch_team(const Prm<T>& P, const LV& L, int i, int j, bool ok) {
  const int q = threadIdx.x & 3;
  const bool open = q == 0 ? (L.px || i > 1) : q == 1 ? (L.px || i < L.m1) : q == 2 ? j > 1 : j < L.m2;
  const int k0 = L.at(i, j);
  const int nq = k0 + (q == 0 ? -1 : q == 1 ? 1 : q == 2 ? -L.pitch : L.pitch);
  ChRows<T> R = ch_team_rows<T, Form>(P, L, i, j, q, open, rho_pair<T, Form>(P, L, k0),
                                      rho_pair<T, Form>(P, L, nq));
  T idet = qrcp(R.J11 * R.J22 - R.J12 * R.J21);
  T dc = (R.J22 * R.Rc - R.J12 * R.Rm) * idet;
  T dm = (R.J11 * R.Rm - R.J21 * R.Rc) * idet;
  if (ok && q == 0) {
    int k = L.at(i, j);
    const bool ghosts = has_ghosts(L, i, j);
    const T cnew = L.c[k] - dc, mnew = L.mu[k] - dm;
    put_cell(L, L.c, i, j, ghosts, cnew);
    if constexpr (!std::is_same<Form, ErrForm>::value)
      put_cell(L, L.rhoc, i, j, ghosts, rho_of(P, cnew));
    put_cell(L, L.mu, i, j, ghosts, mnew);
  }
}

// per-level CH launch with four lanes per cell (colour (i + j) % 2, packed)
template <typename T, class Form>
__global__ void __launch_bounds__(64, 4) k_ch_team(Prm<T> P, Lv<T> L, int colour) {
  pdl_enter();
  int n = L.crow.d * L.m2;
  int t = blockIdx.x * 64 + threadIdx.x;
  if ((t & ~31) >= 4 * n) return;  // warp-uniform
  int i = 1, j = 1;
  bool ok = (t >> 2) < n && ch_slot_cell(L, colour, t >> 2, i, j);
  if (!ok) i = j = 1;
  ch_team<T, Form>(P, L, i, j, ok);
}

// --------------------------------------------------------------------------
// Vanka step 2 of Sec. 7.1: exact solve of the 5x5 block of cell (i,j):
// unknowns (u_W, u_E, v_S, v_N, p), equations (N_u W, N_u E, N_v S, N_v N, N_p).
// Colours: (i + 2j) % 5 (walls in x) or (2i + j) % 8 (periodic x).
// --------------------------------------------------------------------------
// The 5x5 Vanka system of cell (i,j): A = Jacobian of (N_u W, N_u E, N_v S,
// N_v N, N_p) in (u_W, u_E, v_S, v_N, p), b = residuals N - f; rows and
// columns of wall edges (act = false) replaced by the identity.  X: the cell's
// densities on an error level (else unused)
template <typename T, class Form, class LV>
__device__ __forceinline__ void vanka_system(const Prm<T>& P, const LV& L, int i, int j,
                                             const ErrCell<T>* X, T (&A)[5][5], T (&b)[5],
                                             bool (&act)[5]) {
  const int W = L.pitch;
  const T ih = L.ih;
  auto vis = L.visn;
  int k = L.at(i, j);
  int eW = (L.px && i == 1) ? L.m1 : i - 1;
  int kW = L.at(eW, j);
  act[0] = L.px || i > 1;
  act[1] = L.px || i < L.m1;
  act[2] = j > 1;
  act[3] = j < L.m2;
  act[4] = true;
#pragma unroll
  for (int r = 0; r < 5; ++r)
#pragma unroll
    for (int c = 0; c < 5; ++c) A[r][c] = T(0);
  // The rows W, E, S, N sit at these edges.  A periodic cell of column 1 has its
  // west edge as unknown m1, at kW; edge 0 holds its copy, of the coefficients
  // too, and at k - 1 the row shares its values with the other rows.  Only the
  // right-hand side is kept on kW alone.
  const int ke[4] = {k - 1, k, k - W, k};
  const T f[4] = {L.fu[kW], L.fu[k], L.fv[k - W], L.fv[k]};
  const T gt = (j == L.m2) ? T(2) : T(1), gb = (j == 1) ? T(2) : T(1);
  const T ge = (!L.px && i == L.m1) ? T(2) : T(1), gw = (!L.px && i == 1) ? T(2) : T(1);
  const T v3 = vis[k] * L.k.v3;
  T rows[4];  // N of each row, evaluated on wall edges too (padded arrays), then discarded
  if constexpr (std::is_same<Form, ErrForm>::value) {
    const int nb[4] = {2, 1, 4, 3};  // the edge's other cell
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const T rs = X->r[0] + X->r[nb[q]], ds = X->dr[0] + X->dr[nb[q]];
      A[q][q] = err_diag(L, q >> 1, ke[q], rs, q < 2 ? gt : ge, q < 2 ? gb : gw);
      rows[q] = err_row(P, L, q >> 1, ke[q], rs, ds);
    }
    // the coupling of a pair's edges is the stencil's entry for the other one
    A[0][1] = L.aPu[ke[0]];
    A[1][0] = L.aMu[ke[1]];
    A[2][3] = L.aPv[ke[2]];
    A[3][2] = L.aMv[ke[3]];
  } else {
    // density sums on the four edges
    const T rk = Form::rho(P, L, k);
    const T rs[4] = {Form::rho(P, L, k - 1) + rk, rk + Form::rho(P, L, k + 1),
                     Form::rho(P, L, k - W) + rk, rk + Form::rho(P, L, k + W)};
    constexpr bool PROJ = std::is_same<Form, ProjForm>::value;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      A[q][q] = L.pair(q >> 1, L.Dgu, L.Dgv)[ke[q]] + L.k.qidt * rs[q];  // per-step coefficients
      rows[q] = full_mom_row<PROJ>(L, q >> 1, ke[q], rs[q]);
    }
    const T v1 = vis[k] * L.k.v1, sx = L.k.hih * L.Sx[k], sy = L.k.hih * L.Sy[k];
    A[0][1] = sx - v1 - v3;
    A[1][0] = -sx - v1 - v3;
    A[2][3] = sy - v1 - v3;
    A[3][2] = -sy - v1 - v3;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    b[q] = act[q] ? rows[q] - f[q] : T(0);
    const int o = q < 2 ? 2 : 0;  // the couplings to the other direction's edges
    A[q][o] = (q & 1) ? -v3 : v3;
    A[q][o + 1] = (q & 1) ? v3 : -v3;
    A[q][4] = (q & 1) ? -L.k.ihM : L.k.ihM;
  }
  {
    auto mob = L.mobn;
    bool wall[4] = {!L.px && i == L.m1, !L.px && i == 1, j == L.m2, j == 1};
    const int off[4] = {1, -1, W, -W};
    T sm = 0;
#pragma unroll
    for (int f = 0; f < 4; ++f)
      if (!wall[f]) sm += mob[k] + mob[k + off[f]];
    A[4][0] = -ih;
    A[4][1] = ih;
    A[4][2] = -ih;
    A[4][3] = ih;
    A[4][4] = L.k.a2dif * sm;
  }
  if constexpr (std::is_same<Form, ProjForm>::value) b[4] = T(0);  // the 4x4 block has no p row
  else b[4] = (L.u[k] - L.u[k - 1] + L.v[k] - L.v[k - W]) * ih - L.k.adif * flux_sum(P, L, k) - L.fp[k];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (!act[q]) {
#pragma unroll
      for (int c = 0; c < 5; ++c) { A[q][c] = T(0); A[c][q] = T(0); }
      A[q][q] = T(1);
    }
}

// Exact solve of the Vanka system A d = b by its structure.  The velocity block
// is A_vv = B + v3 w w^T: every coupling between an x-edge and a y-edge of the
// cell is +-v3 (the grad-div term), w = (1, -1, 1, -1) on active edges and 0 on
// wall edges, and B is block-diagonal (the x pair and the y pair).  The
// pressure column is a w (a = 1/(M h)) and the pressure row -w/h.  With
// y = B^-1 b_v, z = B^-1 w, s = w.z, t = w.y, g = 1/(1 + v3 s)
// (Sherman-Morrison), p = (b_p + t g/h)/(A_pp + a s g/h) and
// d_v = y - z g (v3 t + a p): two 2x2 solves and three divisions in place of
// 5x5 elimination.  B is diagonally dominant and s, g > 0, so no pivoting.
// NP = 5 solves the full system, NP = 4 the velocity block alone.
template <typename T, int NP>
__device__ __forceinline__ void solve_vanka(const T (&A)[5][5], T (&b)[5], const bool (&act)[5],
                                            T v3, T a, T ih, T iha) {
  // w_q is +1, -1 or 0, so the products with w are selections
  T y[4], z[4];
#pragma unroll
  for (int blk = 0; blk < 4; blk += 2) {
    const int p0 = blk, p1 = blk + 1;
    const bool a0 = act[p0], a1 = act[p1];
    // B = A_vv - v3 w w^T on this pair: w_p0 w_p0 = a0, w_p1 w_p1 = a1, w_p0 w_p1 = -(a0 a1)
    T B00 = a0 ? A[p0][p0] - v3 : A[p0][p0];
    T B11 = a1 ? A[p1][p1] - v3 : A[p1][p1];
    T B01 = (a0 && a1) ? A[p0][p1] + v3 : A[p0][p1];
    T B10 = (a0 && a1) ? A[p1][p0] + v3 : A[p1][p0];
    T idet = qrcp(B00 * B11 - B01 * B10);
    y[p0] = (B11 * b[p0] - B01 * b[p1]) * idet;
    y[p1] = (B00 * b[p1] - B10 * b[p0]) * idet;
    // z = B^-1 w with w_p0 = a0 ? 1 : 0, w_p1 = a1 ? -1 : 0
    T zn0 = (a0 ? B11 : T(0)) + (a1 ? B01 : T(0));
    T zn1 = -((a1 ? B00 : T(0)) + (a0 ? B10 : T(0)));
    z[p0] = zn0 * idet;
    z[p1] = zn1 * idet;
  }
  // inactive entries of y and z are 0 (identity rows, b = 0, w = 0)
  T sdot = (z[0] - z[1]) + (z[2] - z[3]);
  T tdot = (y[0] - y[1]) + (y[2] - y[3]);
  T g = qrcp(T(1) + v3 * sdot);
  T pr = T(0);
  const T tg = tdot * g;
  if constexpr (NP == 5) pr = (b[4] + ih * tg) * qrcp(A[4][4] + iha * (sdot * g));
  T f = v3 * tg;
  if constexpr (NP == 5) f += (a * g) * pr;
#pragma unroll
  for (int q = 0; q < 4; ++q) b[q] = y[q] - z[q] * f;
  if constexpr (NP == 5) b[4] = pr;
}

template <typename T, class Form, class LV>
__device__ __forceinline__ void vanka_cell(const Prm<T>& P, const LV& L, int i, int j, T omega) {
  T A[5][5], b[5];
  bool act[5];
  ErrCell<T> X;
  if constexpr (std::is_same<Form, ErrForm>::value) X = err_cell(P, L, L.at(i, j));
  vanka_system<T, Form>(P, L, i, j, &X, A, b, act);
  const int W = L.pitch;
  int k = L.at(i, j);
  solve_vanka<T, 5>(A, b, act, L.visn[k] * L.k.v3, L.k.ihM, L.ih, L.k.ihaM);
  int eW = (L.px && i == 1) ? L.m1 : i - 1;
  int kW = L.at(eW, j);
  // every old value is read before the first store: a load behind a store that
  // may alias it waits its full latency, once per value
  const bool ghosts = has_ghosts(L, i, j);
  const T w = L.u[kW] - omega * b[0], e = L.u[k] - omega * b[1], so = L.v[k - W] - omega * b[2],
          n = L.v[k] - omega * b[3], pn = L.p[k] - omega * b[4];
  put_edges(L, i, j, ghosts, act, w, e, so, n);
  put_cell(L, L.p, i, j, ghosts, pn);
}

// Exact solve of the coupled 7x7 system of coupled_cell by blocks.  Its NS part
// A[2..6][2..6] is a Vanka block (see solve_vanka): it is factored once and
// applied to three right-hand sides, b_NS and the two columns through which c
// and mu enter the NS rows.  What remains for (dc, dmu) is the 2x2 Schur
// complement S = J_CH - C (A_NS^-1 C'), solved directly; the NS unknowns follow
// by back substitution.  Row 1 (N_mu) does not involve u, v or p, so its
// coupling entries are zero and its Schur row is that of J_CH.
template <typename T>
__device__ __forceinline__ void solve_coupled7(const T (&A)[7][7], T (&b)[7], const bool (&act)[5],
                                               T v3, T a, T ih, T iha) {
  T B00[2], B01[2], B10[2], B11[2], idet[2], z[4];
#pragma unroll
  for (int blk = 0; blk < 2; ++blk) {
    const int p0 = 2 * blk, p1 = p0 + 1;
    const bool a0 = act[p0], a1 = act[p1];
    B00[blk] = a0 ? A[2 + p0][2 + p0] - v3 : A[2 + p0][2 + p0];
    B11[blk] = a1 ? A[2 + p1][2 + p1] - v3 : A[2 + p1][2 + p1];
    B01[blk] = (a0 && a1) ? A[2 + p0][2 + p1] + v3 : A[2 + p0][2 + p1];
    B10[blk] = (a0 && a1) ? A[2 + p1][2 + p0] + v3 : A[2 + p1][2 + p0];
    idet[blk] = qrcp(B00[blk] * B11[blk] - B01[blk] * B10[blk]);
    z[p0] = ((a0 ? B11[blk] : T(0)) + (a1 ? B01[blk] : T(0))) * idet[blk];
    z[p1] = -((a1 ? B00[blk] : T(0)) + (a0 ? B10[blk] : T(0))) * idet[blk];
  }
  const T sdot = (z[0] - z[1]) + (z[2] - z[3]);
  const T g = qrcp(T(1) + v3 * sdot);
  const T iden = qrcp(A[6][6] + iha * (sdot * g)), ga = g * a;
  // x = A_NS^-1 r for a right-hand side r over (u_W, u_E, v_S, v_N, p)
  auto apply = [&](const T (&r)[5], T (&x)[5]) {
    T y[4];
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
      const int p0 = 2 * blk, p1 = p0 + 1;
      y[p0] = (B11[blk] * r[p0] - B01[blk] * r[p1]) * idet[blk];
      y[p1] = (B00[blk] * r[p1] - B10[blk] * r[p0]) * idet[blk];
    }
    T t = (y[0] - y[1]) + (y[2] - y[3]);
    T tg = t * g;
    T pr = (r[4] + ih * tg) * iden;
    T f = v3 * tg + ga * pr;
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = y[q] - z[q] * f;
    x[4] = pr;
  };
  T r0[5], r1[5], r2[5], X0[5], X1[5], X2[5];
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    r0[m] = b[2 + m];
    r1[m] = A[2 + m][0];
    r2[m] = A[2 + m][1];
  }
  apply(r0, X0);
  apply(r1, X1);
  apply(r2, X2);
  T S00 = A[0][0], S01 = A[0][1], rhs0 = b[0];
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    S00 -= A[0][2 + m] * X1[m];
    S01 -= A[0][2 + m] * X2[m];
    rhs0 -= A[0][2 + m] * X0[m];
  }
  const T S10 = A[1][0], S11 = A[1][1], rhs1 = b[1];
  T id2 = qrcp(S00 * S11 - S01 * S10);
  T dc = (S11 * rhs0 - S01 * rhs1) * id2;
  T dm = (S00 * rhs1 - S10 * rhs0) * id2;
  b[0] = dc;
  b[1] = dm;
#pragma unroll
  for (int m = 0; m < 5; ++m) b[2 + m] = X0[m] - X1[m] * dc - X2[m] * dm;
}

// Coupled block (an option; the paper's smoother keeps the two blocks
// separate): one Newton step on the 7x7 system of (N_c, N_mu, N_u W, N_u E,
// N_v S, N_v N, N_p) in (c, mu, u_W, u_E, v_S, v_N, p).  It adds to the 2x2 CH
// and 5x5 Vanka blocks the couplings the separate smoothers treat explicitly:
// the CH advection (e1e2) and (alpha/Pe) grad.(A m grad p) in N_c, the
// (alpha/Pe) grad.(A m grad mu) term of N_p, and the rho(c) and surface-tension
// (e1e1) terms of the momentum rows.
template <typename T, class Form, class LV>
__device__ __forceinline__ void coupled_cell(const Prm<T>& P, const LV& L, int i, int j, T omega) {
  T A5[5][5], b5[5], J2[2][2], R2[2];
  bool act[5];
  ErrCell<T> X;
  if constexpr (std::is_same<Form, ErrForm>::value) {
    X = err_cell(P, L, L.at(i, j));
    ch_system_err(P, L, i, j, X, J2, R2);
  } else {
    ch_system<T, Form>(P, L, i, j, J2, R2);
  }
  vanka_system<T, Form>(P, L, i, j, &X, A5, b5, act);
  T A[7][7], b[7];
#pragma unroll
  for (int r = 0; r < 7; ++r)
#pragma unroll
    for (int c = 0; c < 7; ++c) A[r][c] = T(0);
#pragma unroll
  for (int r = 0; r < 5; ++r) {
    b[2 + r] = b5[r];
#pragma unroll
    for (int c = 0; c < 5; ++c) A[2 + r][2 + c] = A5[r][c];
  }
  A[0][0] = J2[0][0];
  A[0][1] = J2[0][1];
  A[1][0] = J2[1][0];
  A[1][1] = J2[1][1];
  b[0] = R2[0];
  b[1] = R2[1];
  const int W = L.pitch;
  int k = L.at(i, j);
  int eW = (L.px && i == 1) ? L.m1 : i - 1;
  int kW = L.at(eW, j);
  auto rn = L.rhon; auto mob = L.mobn;
  bool wall[4] = {!L.px && i == L.m1, !L.px && i == 1, j == L.m2, j == 1};
  const int off[4] = {1, -1, W, -W};
  T sm = T(0);
#pragma unroll
  for (int f = 0; f < 4; ++f)
    if (!wall[f]) sm += mob[k] + mob[k + off[f]];
  const T rho = J2[1][1], drho = -P.alpha * rho * rho;  // d N_mu / d mu is rho(c)
  // rho^n D c^n / 2 at the four faces of the cell, as in (e1e2) and (e1e1)
  T gW = rn[k - 1] * L.Tx[k - 1];
  T gE = rn[k + 1] * L.Tx[k];
  T gS = rn[k - W] * L.Ty[k - W];
  T gN = rn[k + W] * L.Ty[k];
  T diffc = L.k.adif * sm;
  A[0][2] = gW;
  A[0][3] = gE;
  A[0][4] = gS;
  A[0][5] = gN;
  A[0][6] = diffc;
  T half_idt = T(0.25) * drho * P.idt;  // d/dc of (A rho(c) - A rho^n) x / (2 dt), per edge
  A[2][0] = half_idt * Form::val_u(L, k - 1);
  A[3][0] = half_idt * Form::val_u(L, k);
  A[4][0] = half_idt * Form::val_v(L, k - W);
  A[5][0] = half_idt * Form::val_v(L, k);
  A[2][1] = -gW * P.iM;
  A[3][1] = -gE * P.iM;
  A[4][1] = -gS * P.iM;
  A[5][1] = -gN * P.iM;
  A[6][1] = diffc;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (!act[q]) {
#pragma unroll
      for (int c = 0; c < 7; ++c) {
        A[2 + q][c] = T(0);
        A[c][2 + q] = T(0);
      }
      A[2 + q][2 + q] = T(1);
    }
  solve_coupled7<T>(A, b, act, L.visn[k] * L.k.v3, L.k.ihM, L.ih, L.k.ihaM);
  const bool ghosts = has_ghosts(L, i, j);  // (old values first, as in vanka_cell)
  const T cnew = L.c[k] - omega * b[0], mnew = L.mu[k] - omega * b[1];
  const T w = L.u[kW] - omega * b[2], e = L.u[k] - omega * b[3], so = L.v[k - W] - omega * b[4],
          n = L.v[k] - omega * b[5], pn = L.p[k] - omega * b[6];
  put_cell(L, L.c, i, j, ghosts, cnew);
  if constexpr (!std::is_same<Form, ErrForm>::value)
    put_cell(L, L.rhoc, i, j, ghosts, rho_of(P, cnew));
  put_cell(L, L.mu, i, j, ghosts, mnew);
  put_edges(L, i, j, ghosts, act, w, e, so, n);
  put_cell(L, L.p, i, j, ghosts, pn);
}

// per-level smoother launches: one thread per cell of the colour, packed into
// 64-thread blocks so that a level's warps spread over many SMs (on the FP64
// pipe a warp costs the same with 1 or 32 lanes busy).  The launch bounds ask for
// four blocks an SM: without them the compiler keeps these kernels at 48 to 80
// registers and issues a visit's 60 to 110 loads in batches, each an exposed L2
// round trip; with them all are in flight (FP32 coupled visits 8.2 -> 4.4 us a
// colour on small levels, 9.9 -> 6.1 us on 448x448).  Eight blocks an SM measured
// slower (1024x4096 mixed 83.6 against 78.5 ms a step), two the same.
constexpr int SNT = 64;

template <typename T, class Form>
__global__ void __launch_bounds__(SNT, 4) k_vanka(Prm<T> P, Lv<T> L, int colour, T omega) {
  pdl_enter();
  ColourSlots cs = vanka_slots(L, colour);
  int t = blockIdx.x * SNT + threadIdx.x;
  int i, j;
  if (t >= cs.n || !vanka_slot_cell(L, colour, cs, t, i, j)) return;
  vanka_cell<T, Form>(P, L, i, j, omega);
}

template <typename T, class Form>
__global__ void __launch_bounds__(SNT, 4) k_coupled(Prm<T> P, Lv<T> L, int colour, T omega) {
  pdl_enter();
  ColourSlots cs = vanka_slots(L, colour);
  int t = blockIdx.x * SNT + threadIdx.x;
  int i, j;
  if (t >= cs.n || !vanka_slot_cell(L, colour, cs, t, i, j)) return;
  coupled_cell<T, Form>(P, L, i, j, omega);
}

// --------------------------------------------------------------------------
// projection method (Sec. 7.2): the intermediate-velocity block, pressure
// Gauss-Seidel, the projected velocity and the projection dissipation
// --------------------------------------------------------------------------
// step 2: exact solve of the 4x4 block of the intermediate velocities
// (ut_W, ut_E, vt_S, vt_N) of cell (i,j) in the rows of (pj-num-mx)
template <typename T, class Form, class LV>
__device__ __forceinline__ void vanka4_cell(const Prm<T>& P, const LV& L, int i, int j, T omega) {
  T A5[5][5], b5[5];
  bool act[5];
  vanka_system<T, Form>(P, L, i, j, (const ErrCell<T>*)nullptr, A5, b5, act);
  const int W = L.pitch;
  int k = L.at(i, j);
  solve_vanka<T, 4>(A5, b5, act, L.visn[k] * L.k.v3, L.k.ihM, L.ih, L.k.ihaM);
  const T(&b)[5] = b5;
  int eW = (L.px && i == 1) ? L.m1 : i - 1;
  int kW = L.at(eW, j);
  const bool ghosts = has_ghosts(L, i, j);
  const T w = L.u[kW] - omega * b[0], e = L.u[k] - omega * b[1], so = L.v[k - W] - omega * b[2],
          n = L.v[k] - omega * b[3];
  put_edges(L, i, j, ghosts, act, w, e, so, n);
}

template <typename T, class Form>
__global__ void __launch_bounds__(SNT, 4) k_vanka4(Prm<T> P, Lv<T> L, int colour, T omega) {
  pdl_enter();
  ColourSlots cs = vanka_slots(L, colour);
  int t = blockIdx.x * SNT + threadIdx.x;
  int i, j;
  if (t >= cs.n || !vanka_slot_cell(L, colour, cs, t, i, j)) return;
  vanka4_cell<T, Form>(P, L, i, j, omega);
}

// step 3: Gauss-Seidel on (pj-num-mass) for p_ij.  The row is affine in p_ij:
// u^{n+1} on an open face carries -dt/(M h A rho(c)) times the pressure of each
// adjacent cell, plus the diffusion term (alpha^2/Pe) A m / h^2.
template <typename T, class LV>
__device__ __forceinline__ void pgs_cell(const Prm<T>& P, const LV& L, int i, int j) {
  const int W = L.pitch;
  int k = L.at(i, j);
  auto rc = L.rhoc;
  T rk = rc[k];
  const T rq[4] = {rc[k + 1], rc[k - 1], rc[k + W], rc[k - W]};
  T w[4];
  proj_faces(P, L, i, j, rk, rq, w);
  T R = opp_p_w(L, w, flux_sum(P, L, k)) - L.fp[k];
  const bool wall[4] = {!L.px && i == L.m1, !L.px && i == 1, j == L.m2, j == 1};
  const int off[4] = {1, -1, W, -W};
  T d = T(0);
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    if (wall[f]) continue;
    int q = k + off[f];
    d += L.k.pdiv * qrcp(rk + rq[f]) + L.k.a2dif * (L.mobn[k] + L.mobn[q]);
  }
  put_cell(L, L.p, i, j, has_ghosts(L, i, j), L.p[k] - R * qrcp(d));
}

// pgs_cell by a team of four lanes (lane & 3 = q: face W, E, S, N): lane q
// takes u^{n+1} at face q, its share of the mass row and of the row's
// derivative in p_ij; butterflies add them; lane 0 stores.
template <typename T, class LV>
__device__ __forceinline__ void pgs_team(const Prm<T>& P, const LV& L, int i, int j, bool ok) {
  const int W = L.pitch;
  const int q = threadIdx.x & 3;
  const bool open = q == 0 ? (L.px || i > 1) : q == 1 ? (L.px || i < L.m1) : q == 2 ? j > 1 : j < L.m2;
  int k = L.at(i, j);
  const int nq = k + (q == 0 ? -1 : q == 1 ? 1 : q == 2 ? -W : W);
  T rk = L.rhoc[k], rq = L.rhoc[nq];
  T wq = proj_face_team(P, L, k, q, open, rk, rq);
  T am = L.mobn[nq] + L.mobn[k];
  T sdiv = team_sum<T>((q & 1) ? wq : -wq);
  T sflux = team_sum<T>(am * ((L.mu[nq] - L.mu[k]) + P.alpha * (L.p[nq] - L.p[k])));
  T sd = team_sum<T>(open ? L.k.pdiv * qrcp(rk + rq) + L.k.a2dif * am : T(0));
  T R = sdiv * L.ih - L.k.adif * sflux - L.fp[k];
  const T pn = L.p[k] - R * qrcp(sd);
  if (ok && q == 0) put_cell(L, L.p, i, j, has_ghosts(L, i, j), pn);
}

template <typename T>
__global__ void __launch_bounds__(64, 4) k_pgs_team(Prm<T> P, Lv<T> L, int colour) {
  pdl_enter();
  int n = L.crow.d * L.m2;
  int t = blockIdx.x * 64 + threadIdx.x;
  if ((t & ~31) >= 4 * n) return;  // warp-uniform
  int i = 1, j = 1;
  bool ok = (t >> 2) < n && ch_slot_cell(L, colour, t >> 2, i, j);
  if (!ok) i = j = 1;
  pgs_team<T>(P, L, i, j, ok);
}

// cells of colour (i + j) % 2 == colour, packed as in k_ch
template <typename T>
__global__ void __launch_bounds__(64, 4) k_pgs(Prm<T> P, Lv<T> L, int colour) {
  pdl_enter();
  int t = blockIdx.x * 64 + threadIdx.x, i, j;
  if (t >= L.crow.d * L.m2 || !ch_slot_cell(L, colour, t, i, j)) return;
  pgs_cell<T>(P, L, i, j);
}

// u^{n+1} on the x-edges i = 0..m1 (rows 1..m2) and v^{n+1} on the y-edges
// j = 0..m2 (columns 1..m1), into uo, vo (level layout); ghosts are filled after
template <typename T>
__global__ void k_proj_velocity(Prm<T> P, Lv<T> L, T* uo, T* vo) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x;
  int j = blockIdx.y * BY + threadIdx.y;
  if (i > L.m1 || j > L.m2) return;
  int k = L.at(i, j);
  if (j >= 1) uo[k] = proj_u(P, L, i, j);
  if (i >= 1) vo[k] = proj_v(P, L, i, j);
}

// the projection method's extra dissipation, 1/2 ||sqrt(rho(c)) (u^{n+1} - ut)||^2
// in the cell-averaged form of the kinetic energy; per cell before the h^2/2
template <typename T>
__global__ void k_proj_diss(Prm<T> P, Lv<T> L, const T* uo, const T* vo, double* part) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x + 1;
  int j = blockIdx.y * BY + threadIdx.y + 1;
  double val[1] = {0.0};
  if (i <= L.m1 && j <= L.m2) {
    const int W = L.pitch;
    int k = L.at(i, j);
    double r = 1.0 / ((double)P.ia * (double)L.c[k] + (double)P.ib);
    double a = (double)uo[k] - (double)L.u[k], b = (double)uo[k - 1] - (double)L.u[k - 1];
    double c = (double)vo[k] - (double)L.v[k], d = (double)vo[k - W] - (double)L.v[k - W];
    val[0] = r * (0.5 * (a * a + b * b) + 0.5 * (c * c + d * d));
  }
  block_sum_store<1>(val, part, 0);
}

// --------------------------------------------------------------------------
// ghost filling (App. A.6): every ghost entry computed from interior entries
// --------------------------------------------------------------------------
__device__ __forceinline__ int xsrc_cell(int I, int m1, int px) {
  if (I == 0) return px ? m1 : 1;
  if (I == m1 + 1) return px ? 1 : m1;
  return I;
}

// band: I = -1..m1+1 on rows J in {-1, 0, 1?}... we enumerate a 4-wide frame
__device__ __forceinline__ bool frame_pos(int t, int m1, int m2, int& I, int& J) {
  int NX = m1 + 3, NY = m2 + 3;
  if (t < 4 * NX) {
    int r = (t >= NX) + (t >= 2 * NX) + (t >= 3 * NX);
    I = t - r * NX - 1;
    J = r < 2 ? r - 1 : m2 + r - 2;  // rows -1, 0, m2, m2+1
    return true;
  }
  t -= 4 * NX;
  if (t < 4 * NY) {
    int cidx = (t >= NY) + (t >= 2 * NY) + (t >= 3 * NY);
    J = t - cidx * NY - 1;
    I = cidx < 2 ? cidx - 1 : m1 + cidx - 2;  // columns -1, 0, m1, m1+1
    return true;
  }
  return false;
}

template <class LV, class A>
__device__ __forceinline__ void fill_cell_ghost(const LV& L, A a, int I, int J) {
  typedef typename LV::real T;
  if (I < 0 || J < 0) return;
  bool gx = (I == 0 || I == L.m1 + 1), gy = (J == 0 || J == L.m2 + 1);
  if (!gx && !gy) return;
  int si = xsrc_cell(I, L.m1, L.px);
  int sj = J == 0 ? 1 : (J == L.m2 + 1 ? L.m2 : J);
  a[L.at(I, J)] = a[L.at(si, sj)];
}

template <class LV, class A>
__device__ __forceinline__ typename LV::real u_interior_or_zero(const LV& L, A a, int I, int J) {
  typedef typename LV::real T;
  // value of u(I, J) for J in 1..m2 after applying the x rule
  if (L.px) {
    int s = I;
    if (I == 0) s = L.m1;
    else if (I == -1) s = L.m1 - 1;
    else if (I == L.m1 + 1) s = 1;
    return a[L.at(s, J)];
  }
  if (I <= 0 || I >= L.m1) return T(0);
  return a[L.at(I, J)];
}

template <class LV, class A>
__device__ __forceinline__ void fill_u_ghost(const LV& L, A a, int I, int J) {
  typedef typename LV::real T;
  if (J < 0) return;
  bool xg = L.px ? (I == 0 || I == -1 || I == L.m1 + 1) : (I <= 0 || I >= L.m1);
  bool yg = (J == 0 || J == L.m2 + 1);
  if (!xg && !yg) return;
  if (yg) {
    int sj = J == 0 ? 1 : L.m2;
    a[L.at(I, J)] = -u_interior_or_zero(L, a, I, sj);
  } else {
    a[L.at(I, J)] = u_interior_or_zero(L, a, I, J);
  }
}

template <class LV, class A>
__device__ __forceinline__ typename LV::real v_interior_or_zero(const LV& L, A a, int I, int J) {
  typedef typename LV::real T;
  // value of v(I, J) for I in 1..m1 after applying the y (wall) rule
  if (J <= 0 || J >= L.m2) return T(0);
  return a[L.at(I, J)];
}

template <class LV, class A>
__device__ __forceinline__ void fill_v_ghost(const LV& L, A a, int I, int J) {
  typedef typename LV::real T;
  if (I < 0) return;
  bool xg = (I == 0 || I == L.m1 + 1);
  bool yg = (J <= 0 || J >= L.m2);
  if (!xg && !yg) return;
  if (xg) {
    int si = xsrc_cell(I, L.m1, L.px);
    T s = v_interior_or_zero(L, a, si, J);
    a[L.at(I, J)] = L.px ? s : -s;
  } else {
    a[L.at(I, J)] = T(0);
  }
}

template <typename T>
__global__ void __launch_bounds__(NT, 2) k_bc_unknowns(Lv<T> L) {
  pdl_enter();
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  int I, J;
  if (!frame_pos(t, L.m1, L.m2, I, J)) return;
  fill_cell_ghost(L, L.c, I, J);
  if (L.rhoc) fill_cell_ghost(L, L.rhoc, I, J);
  fill_cell_ghost(L, L.mu, I, J);
  fill_cell_ghost(L, L.p, I, J);
  fill_u_ghost(L, L.u, I, J);
  fill_v_ghost(L, L.v, I, J);
}

template <typename T>
__global__ void __launch_bounds__(NT, 2) k_bc_frozen(Lv<T> L) {
  pdl_enter();
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  int I, J;
  if (!frame_pos(t, L.m1, L.m2, I, J)) return;
  fill_cell_ghost(L, L.cn, I, J);
  fill_u_ghost(L, L.un, I, J);
  fill_v_ghost(L, L.vn, I, J);
}

// rho(c^n), m(c^n), mu(c^n) on the whole ghosted cell range; G(c^n) inside
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_frozen_derived(Prm<T> P, Lv<T> L) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x;
  int j = blockIdx.y * BY + threadIdx.y;
  if (i > L.m1 + 1 || j > L.m2 + 1) return;
  int k = L.at(i, j);
  T c = L.cn[k];
  L.rhon[k] = rho_of(P, c);
  L.mobn[k] = mob_of(P, c);
  L.visn[k] = visc_of(P, c);
  if (i >= 1 && i <= L.m1 && j >= 1 && j <= L.m2) L.Gn[k] = G_h2(L.cn, k, L.pitch) * L.ih2;
}

// frozen coefficients of (pm-num-mx): cells and vertices (needs rho^n, mu(c^n), ghosts)
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_frozen_coef1(Lv<T> L) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x;
  int j = blockIdx.y * BY + threadIdx.y;
  if (i > L.m1 + 1 || j > L.m2 + 1) return;
  const int W = L.pitch;
  int k = L.at(i, j);
  auto rn = L.rhon; auto vis = L.visn; auto un = L.un; auto vn = L.vn; auto cn = L.cn;
  L.Sx[k] = rn[k] * T(0.5) * (un[k] + un[k - 1]);   // cell (i,j)
  L.Sy[k] = rn[k] * T(0.5) * (vn[k] + vn[k - W]);
  if (i <= L.m1 && j <= L.m2) {  // vertex (i+1/2, j+1/2), edges (i+1/2, j), (i, j+1/2)
    T Ar = T(0.25) * (rn[k] + rn[k + 1] + rn[k + W] + rn[k + 1 + W]);
    L.Qx[k] = Ar * T(0.5) * (vn[k + 1] + vn[k]);
    L.Qy[k] = Ar * T(0.5) * (un[k + W] + un[k]);
    L.Av[k] = T(0.25) * (vis[k] + vis[k + 1] + vis[k + W] + vis[k + 1 + W]);
    L.Aru[k] = T(0.5) * (rn[k] + rn[k + 1]);
    L.Arv[k] = T(0.5) * (rn[k] + rn[k + W]);
    L.Tx[k] = T(0.5) * (cn[k + 1] - cn[k]) * L.ih;
    L.Ty[k] = T(0.5) * (cn[k + W] - cn[k]) * L.ih;
  }
}

// divergence corrections of (e1e1-2) on edges (needs k_frozen_coef1)
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_frozen_coef2(Lv<T> L) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x;
  int j = blockIdx.y * BY + threadIdx.y;
  if (i > L.m1 || j > L.m2) return;
  const int W = L.pitch;
  int k = L.at(i, j);
  if (j >= 1) L.Dvu[k] = T(0.5) * ((L.Sx[k + 1] - L.Sx[k]) + (L.Qx[k] - L.Qx[k - W])) * L.ih;
  if (i >= 1) L.Dvv[k] = T(0.5) * ((L.Qy[k] - L.Qy[k - 1]) + (L.Sy[k + W] - L.Sy[k])) * L.ih;
}

// The assembled stencil of one momentum row of (pm-num-mx) at edge k (mom_asm):
// s the stride along the edge normal, t across it; S the cell-centred and Q the
// vertex convection coefficients, Tf = D c^n / 2 on the edge, t1 the time
// term's coefficient T1.  With the differences of the row written out,
//   conv = 1/2 h^-1 (S[k+s] (a[k+s] - a) - S[k] (a - a[k-s]) ... )  and
//   visc = -h^-2/Re ((4/3)(vis[k+s] (a[k+s] - a) - vis[k] (a - a[k-s]))
//                    + Av[k] (a[k+t] - a) - Av[k-t] (a - a[k-t])) + cross terms,
// each neighbour's coefficient is the sum of its convective and viscous
// parts, and the edge's own coefficient is minus their sum plus t1.  Wall
// edges keep the undoubled coefficients: the row reads the reflected ghosts.
template <typename T, class LV, class A>
__device__ __forceinline__ void assemble_row(const Prm<T>& P, const LV& L, int k, int s, int t,
                                             T t1, A S, const T* Q, const T* Tf, T* C,
                                             T* aP, T* aM, T* tP, T* tM, T* M0, T* M1) {
  const T* vis = L.visn;
  const T hc = T(0.5) * L.ih, hv = P.iRe * L.ih2, f43 = T(4.0 / 3.0);
  T vl = vis[k], vr = vis[k + s];
  T ap = hc * S[k + s] - f43 * hv * vr;
  T am = -hc * S[k] - f43 * hv * vl;
  T tp = hc * Q[k] - hv * L.Av[k];
  T tm = -hc * Q[k - t] - hv * L.Av[k - t];
  aP[k] = ap;
  aM[k] = am;
  tP[k] = tp;
  tM[k] = tm;
  C[k] = t1 + hc * (-S[k + s] + S[k] - Q[k] + Q[k - t]) +
         hv * (f43 * (vr + vl) + L.Av[k] + L.Av[k - t]);
  M0[k] = -L.rhon[k + s] * Tf[k] * P.iM;
  M1[k] = -L.rhon[k] * Tf[k] * P.iM;
}

// per-step row coefficients of the momentum rows (needs k_frozen_coef2): time =
// x T1 + T0 + A rho(c) x/(2dt) (T0 of the y rows holds gravity, which P carries
// for the primitive method only); Dg = the iterate-independent part of the
// diagonal entry (the whole entry is Dg + A rho(c)/(2dt)), with the reflected
// no-slip ghosts doubling the tangential wall terms (g = 2)
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_frozen_coef3(Prm<T> P, Lv<T> L) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x;
  int j = blockIdx.y * BY + threadIdx.y;
  if (i > L.m1 || j > L.m2) return;
  const int W = L.pitch;
  int k = L.at(i, j);
  auto vis = L.visn;
  const T third = T(1.0 / 3.0);
  if (j >= 1) {  // x-edge (i+1/2, j)
    T Arn = L.Aru[k];
    T gt = (j == L.m2) ? T(2) : T(1), gb = (j == 1) ? T(2) : T(1);
    T t1 = T(0.5) * Arn * P.idt + L.Dvu[k];
    L.T1u[k] = t1;
    L.T0u[k] = -Arn * L.un[k] * P.idt;
    L.Dgu[k] = t1 + T(0.5) * L.ih * (-L.Sx[k + 1] + L.Sx[k] - L.Qx[k] * gt + L.Qx[k - W] * gb) +
               P.iRe * L.ih2 * ((vis[k + 1] + vis[k]) * (T(1) + third) + gt * L.Av[k] + gb * L.Av[k - W]);
    assemble_row(P, L, k, 1, W, t1, L.Sx, L.Qx, L.Tx, L.Cu, L.aPu, L.aMu, L.tPu, L.tMu, L.M0u,
                 L.M1u);
  }
  if (i >= 1) {  // y-edge (i, j+1/2)
    T Arn = L.Arv[k];
    T ge = (!L.px && i == L.m1) ? T(2) : T(1), gw = (!L.px && i == 1) ? T(2) : T(1);
    T t1 = T(0.5) * Arn * P.idt + L.Dvv[k];
    L.T1v[k] = t1;
    L.T0v[k] = -Arn * L.vn[k] * P.idt + P.Fr_inv * Arn;
    L.Dgv[k] = t1 + T(0.5) * L.ih * (-L.Qy[k] * ge + L.Qy[k - 1] * gw - L.Sy[k + W] + L.Sy[k]) +
               P.iRe * L.ih2 * (ge * L.Av[k] + gw * L.Av[k - 1] + (vis[k + W] + vis[k]) * (T(1) + third));
    assemble_row(P, L, k, W, 1, t1, L.Sy, L.Qy, L.Ty, L.Cv, L.aPv, L.aMv, L.tPv, L.tMv, L.M0v,
                 L.M1v);
  }
}

// --------------------------------------------------------------------------
// FAS transfers
// --------------------------------------------------------------------------
// coarse iterate = R x_h (cells: 4-mean; edges: mean of the 2 coincident fine edges)
// with its ghosts, and a copy kept for the correction.  The stores that keep
// ghosts cover all of them but the cells' corners, which no operator reads:
// wall edges and what lies beyond them are zero from the start.
template <typename T, class LV>
__device__ __forceinline__ void restrict_state_cell(const Prm<T>& P, const LV& F, const LV& C,
                                                    int I, int J) {
  int kc = C.at(I, J);
  const bool cell = I >= 1 && J >= 1;
  T a = T(0), b = T(0), d = T(0), u = T(0), v = T(0);
  if (cell) {
    int kf = F.at(2 * I - 1, 2 * J - 1), W = F.pitch;
    a = T(0.25) * (F.c[kf] + F.c[kf + 1] + F.c[kf + W] + F.c[kf + W + 1]);
    b = T(0.25) * (F.mu[kf] + F.mu[kf + 1] + F.mu[kf + W] + F.mu[kf + W + 1]);
    d = T(0.25) * (F.p[kf] + F.p[kf + 1] + F.p[kf + W] + F.p[kf + W + 1]);
  }
  if (J >= 1) {  // u edge (I, J), I = 0..M1
    int kf = F.at(2 * I, 2 * J - 1);
    u = T(0.5) * (F.u[kf] + F.u[kf + F.pitch]);
  }
  if (I >= 1) {  // v edge (I, J), J = 0..M2
    int kf = F.at(2 * I - 1, 2 * J);
    v = T(0.5) * (F.v[kf] + F.v[kf + 1]);
  }
  const bool ghosts = has_ghosts(C, I, J);
  if (cell) {
    put_cell(C, C.c, I, J, ghosts, a);
    if constexpr (LV::has_rho)
      if (C.rhoc) put_cell(C, C.rhoc, I, J, ghosts, rho_of(P, a));
    put_cell(C, C.mu, I, J, ghosts, b);
    put_cell(C, C.p, I, J, ghosts, d);
    C.sc[kc] = a;
    C.smu[kc] = b;
    C.sp[kc] = d;
  }
  if (J >= 1) {
    if (I >= 1 && I <= C.uhi()) {
      if (ghosts) store_u(C, I, J, u);
      else C.u[kc] = u;
    }
    C.su[kc] = u;
  }
  if (I >= 1) {
    if (J >= 1 && J < C.m2) {
      if (ghosts) store_v(C, I, J, v);
      else C.v[kc] = v;
    }
    C.sv[kc] = v;
  }
}

template <class LV>
__device__ __forceinline__ typename LV::real ru_at(const LV& F, int i, int j) {
  typedef typename LV::real T;
  if (F.px) {
    if (i > F.m1) i -= F.m1;
    if (i < 1) i += F.m1;
  } else if (i <= 0 || i >= F.m1) {
    return T(0);
  }
  return F.ru[F.at(i, j)];
}
template <class LV>
__device__ __forceinline__ typename LV::real rv_at(const LV& F, int i, int j) {
  typedef typename LV::real T;
  if (j <= 0 || j >= F.m2) return T(0);
  return F.rv[F.at(i, j)];
}

// coarse right-hand side f_H = R r_h (cells: 4-mean; edges: full weighting),
// to which k_residual<MODE 1> then adds N_H(R x_h)
template <class LV>
__device__ __forceinline__ void restrict_res_cell(const LV& F, const LV& C, int I, int J) {
  typedef typename LV::real T;
  int kc = C.at(I, J);
  int kf = F.at(2 * I - 1, 2 * J - 1), W = F.pitch;
  const T c = T(0.25) * (F.rc[kf] + F.rc[kf + 1] + F.rc[kf + W] + F.rc[kf + W + 1]);
  const T m = T(0.25) * (F.rmu[kf] + F.rmu[kf + 1] + F.rmu[kf + W] + F.rmu[kf + W + 1]);
  const T p = T(0.25) * (F.rp[kf] + F.rp[kf + 1] + F.rp[kf + W] + F.rp[kf + W + 1]);
  T u = T(0), v = T(0);
  if (I <= C.uhi()) {
#pragma unroll
    for (int jj = 0; jj < 2; ++jj) {
      int jf = 2 * J - 1 + jj;
      u += T(0.25) * ru_at(F, 2 * I - 1, jf) + T(0.5) * ru_at(F, 2 * I, jf) +
           T(0.25) * ru_at(F, 2 * I + 1, jf);
    }
  }
  if (J < C.m2) {
#pragma unroll
    for (int ii = 0; ii < 2; ++ii) {
      int ifn = 2 * I - 1 + ii;
      v += T(0.25) * rv_at(F, ifn, 2 * J - 1) + T(0.5) * rv_at(F, ifn, 2 * J) +
           T(0.25) * rv_at(F, ifn, 2 * J + 1);
    }
  }
  C.fc[kc] = c;
  C.fmu[kc] = m;
  C.fp[kc] = p;
  if (I <= C.uhi()) C.fu[kc] = T(0.5) * u;
  if (J < C.m2) C.fv[kc] = T(0.5) * v;
}

// The coarse level's iterate (restrict_state_cell) and right-hand side R r_h in
// one launch, ghosts stored with their cells: three launches before, one of
// them a frame fill of 2 to 6 us (with k_prolong's, 256x512 mixed 20.2 -> 18.1 ms
// for three steps).  Bound by the launch on small levels, by bytes on large.
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_restrict(Prm<T> P, Lv<T> F, Lv<T> C) {
  pdl_enter();
  int I = blockIdx.x * BX + threadIdx.x;
  int J = blockIdx.y * BY + threadIdx.y;
  if (I > C.m1 || J > C.m2) return;
  if (I >= 1 && J >= 1) restrict_res_cell(F, C, I, J);
  restrict_state_cell(P, F, C, I, J);
}

template <typename T>
__global__ void __launch_bounds__(NT, 2) k_restrict_frozen(Lv<T> F, Lv<T> C) {
  pdl_enter();
  int I = blockIdx.x * BX + threadIdx.x;
  int J = blockIdx.y * BY + threadIdx.y;
  if (I > C.m1 || J > C.m2) return;
  int kc = C.at(I, J);
  if (I >= 1 && J >= 1) {
    int kf = F.at(2 * I - 1, 2 * J - 1), W = F.pitch;
    C.cn[kc] = T(0.25) * (F.cn[kf] + F.cn[kf + 1] + F.cn[kf + W] + F.cn[kf + W + 1]);
  }
  if (J >= 1) {
    int kf = F.at(2 * I, 2 * J - 1);
    C.un[kc] = T(0.5) * (F.un[kf] + F.un[kf + F.pitch]);
  }
  if (I >= 1) {
    int kf = F.at(2 * I - 1, 2 * J);
    C.vn[kc] = T(0.5) * (F.vn[kf] + F.vn[kf + 1]);
  }
}

// x_h += P(x_H - saved_H), with the ghosts (as restrict_state_cell): cells
// piecewise constant; edges coincident or linear in the normal direction,
// constant in the tangential direction
template <typename T, class LV>
__device__ __forceinline__ void prolong_cell(const Prm<T>& P, const LV& F, const LV& C, int i,
                                             int j) {
  int k = F.at(i, j);
  int I = (i + 1) >> 1, J = (j + 1) >> 1;
  int kc = C.at(I, J);
  const T c = F.c[k] + (C.c[kc] - C.sc[kc]), mu = F.mu[k] + (C.mu[kc] - C.smu[kc]),
          p = F.p[k] + (C.p[kc] - C.sp[kc]);
  const bool hu = i <= F.uhi(), hv = j < F.m2;
  T u = T(0), v = T(0);
  if (hu) {
    T e;
    if ((i & 1) == 0) {
      int q = C.at(i >> 1, J);
      e = C.u[q] - C.su[q];
    } else {
      int q0 = C.at((i - 1) >> 1, J), q1 = C.at((i + 1) >> 1, J);
      e = T(0.5) * ((C.u[q0] - C.su[q0]) + (C.u[q1] - C.su[q1]));
    }
    u = F.u[k] + e;
  }
  if (hv) {
    T e;
    if ((j & 1) == 0) {
      int q = C.at(I, j >> 1);
      e = C.v[q] - C.sv[q];
    } else {
      int q0 = C.at(I, (j - 1) >> 1), q1 = C.at(I, (j + 1) >> 1);
      e = T(0.5) * ((C.v[q0] - C.sv[q0]) + (C.v[q1] - C.sv[q1]));
    }
    v = F.v[k] + e;
  }
  const bool ghosts = has_ghosts(F, i, j);
  put_cell(F, F.c, i, j, ghosts, c);
  if constexpr (LV::has_rho)
    if (F.rhoc) put_cell(F, F.rhoc, i, j, ghosts, rho_of(P, c));
  put_cell(F, F.mu, i, j, ghosts, mu);
  put_cell(F, F.p, i, j, ghosts, p);
  if (hu) {
    if (ghosts) store_u(F, i, j, u);
    else F.u[k] = u;
  }
  if (hv) {
    if (ghosts) store_v(F, i, j, v);
    else F.v[k] = v;
  }
}

template <typename T>
__global__ void __launch_bounds__(NT, 2) k_prolong(Prm<T> P, Lv<T> F, Lv<T> C) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x + 1;
  int j = blockIdx.y * BY + threadIdx.y + 1;
  if (i > F.m1 || j > F.m2) return;
  prolong_cell(P, F, C, i, j);
}

// --------------------------------------------------------------------------
// the coarse end of a V-cycle in one launch: levels small enough for one SM,
// or for one thread-block cluster of up to 16 SMs, run their smoothing
// colours, residuals, transfers and ghost fills as group-stride loops
// separated by group barriers (__syncthreads(), or the cluster barrier), one
// launch instead of dozens.  Per-cell work is the same device code as the grid
// kernels above, in the same colour order, so the results are the same.
// --------------------------------------------------------------------------
// coarse base X_H = R X_h (cells: 4-mean; edges: 2 coincident fine edges), one
// entry, with the ghosts that the rows read: those of c and rho(c)
template <typename T, class LV>
__device__ __forceinline__ void restrict_base_cell(const Prm<T>& P, const LV& F, const LV& C, int I,
                                                   int J) {
  const int kc = C.at(I, J);
  const bool ghosts = has_ghosts(C, I, J);
  if (I >= 1 && J >= 1) {
    int kf = F.at(2 * I - 1, 2 * J - 1), W = F.pitch;
    const T B = T(0.25) * (F.Bc[kf] + F.Bc[kf + 1] + F.Bc[kf + W] + F.Bc[kf + W + 1]);
    const T m = T(0.25) * (F.Bmu[kf] + F.Bmu[kf + 1] + F.Bmu[kf + W] + F.Bmu[kf + W + 1]);
    const T d = T(0.25) * (F.Bdc[kf] + F.Bdc[kf + 1] + F.Bdc[kf + W] + F.Bdc[kf + W + 1]);
    put_cell(C, C.Bc, I, J, ghosts, B);
    put_cell(C, C.rB, I, J, ghosts, rho_of(P, B));
    C.Bmu[kc] = m;
    C.Bdc[kc] = d;
  }
  // velocities at the edges of the cells, column 0 (periodic x) included
  if (J >= 1) {
    int kf = F.at(2 * I, 2 * J - 1);
    C.Bu[kc] = T(0.5) * (F.Bu[kf] + F.Bu[kf + F.pitch]);
  }
  if (I >= 1) {
    int kf = F.at(2 * I - 1, 2 * J);
    C.Bv[kc] = T(0.5) * (F.Bv[kf] + F.Bv[kf + 1]);
  }
}

// The fused V-cycle runs in one thread block or in one thread-block cluster of
// gridDim.x blocks (the grid is the cluster).  Its loops and colour steps go
// over a rank of the whole group.  Warps are interleaved across the blocks:
// rank = ((warp * blocks + block) * 32 + lane), so the first 4 x blocks warps
// of a colour step sit on distinct SM sub-partitions (warp w of a block runs on
// sub-partition w mod 4), each of which owns one FP64 pipe.  The low five bits
// of the rank are the hardware lane, so four-lane teams stay inside a warp.
// One block: the rank is threadIdx.x and the step barrier is __syncthreads().
// A cluster: the barrier is the hardware cluster barrier, whose release and
// acquire order every block's global-memory writes before the next step's
// reads; every thread of the cluster reaches every barrier.
__device__ __forceinline__ int grp_rank() {
  return (((threadIdx.x >> 5) * gridDim.x + blockIdx.x) << 5) | (threadIdx.x & 31);
}
__device__ __forceinline__ int grp_size() { return gridDim.x * blockDim.x; }
__device__ __forceinline__ void grp_sync() {
  if (gridDim.x == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  }
}

template <typename T>
struct CoarseLevels {
  Lv<T> L[QN_MAX_FUSED_LEVELS];
  int n;
  int base;  // error equation: restrict the base state to L[1..n-1] first
};

// --------------------------------------------------------------------------
// single-block smoothing of the coarse levels.  An FP64 warp instruction
// holds the SM sub-partition's FP64 pipe for about 64 cycles however many of
// its lanes are active, so a colour step on a small level costs (warp
// instructions per visit) x (warps per sub-partition): threads are packed onto
// the cells of the colour, and on the smallest levels four lanes share one
// Vanka block (one edge row each).
// --------------------------------------------------------------------------
// N - f of the momentum row in direction d (0: the x row, unknown u; 1:
// the y row, unknown v) at edge index k: full_mom_row, or err_row for ErrForm, from
// rho(c) of the edge's two cells; kf is the index of its right-hand side.  Both
// directions run the same instructions on different arrays and strides (s
// along the edge normal, t across it).
template <typename T, class Form, class LV>
__device__ __forceinline__ T mom_residual(const Prm<T>& P, const LV& L, int d, int k, int kf,
                                          RhoPair<T> l, RhoPair<T> r) {
  const T f = L.pair(d, L.fu, L.fv)[kf];
  if constexpr (std::is_same<Form, ErrForm>::value)
    return err_row(P, L, d, k, l.r + r.r, l.d + r.d) - f;
  else
    return full_mom_row<std::is_same<Form, ProjForm>::value>(L, d, k, l.r + r.r) - f;
}

// Diagonal entry dq and residual bq = N - f (0 on a wall edge) of momentum row
// q of the Vanka block of cell (i,j), for lane q of a team: direction d (0:
// x-edge, 1: y-edge), edge index ke of the row (its copy at column 0 for a
// periodic west edge) and kf of its right-hand side, rho(c) of the edge's
// cells l and r.
template <typename T, class Form, class LV>
__device__ __forceinline__ void team_row(const Prm<T>& P, const LV& L, int i, int j, int d, int ke,
                                         int kf, RhoPair<T> l, RhoPair<T> r, bool mine, T& dq,
                                         T& bq) {
  if constexpr (std::is_same<Form, ErrForm>::value) {
    T gp = d ? ((!L.px && i == L.m1) ? T(2) : T(1)) : ((j == L.m2) ? T(2) : T(1));
    T gm = d ? ((!L.px && i == 1) ? T(2) : T(1)) : ((j == 1) ? T(2) : T(1));
    dq = err_diag(L, d, ke, l.r + r.r, gp, gm);
  } else {
    dq = L.pair(d, L.Dgu, L.Dgv)[ke] + L.k.qidt * (l.r + r.r);
  }
  bq = mom_residual<T, Form>(P, L, d, ke, kf, l, r);  // wall edges too (padded arrays), then discarded
  if (!mine) bq = T(0);
}
// the couplings b01, b10 of the two edges of direction d of cell k within B
// (the block without its v3 part): (first row, second edge) and the converse
template <typename T, class Form, class LV>
__device__ __forceinline__ void pair_couplings(const LV& L, int d, int k, T vc, T& b01, T& b10) {
  if constexpr (std::is_same<Form, ErrForm>::value) {
    const T v3 = vc * L.k.v3;
    b01 = L.pair(d, L.aPu, L.aPv)[k - (d ? L.pitch : 1)] + v3;
    b10 = L.pair(d, L.aMu, L.aMv)[k] + v3;
  } else {
    const T v1 = vc * L.k.v1, sc = L.k.hih * L.pair(d, L.Sx, L.Sy)[k];
    b01 = sc - v1;
    b10 = -sc - v1;
  }
}

// The structured solve of solve_vanka, split over a team of four lanes.  The
// velocity block is B + v3 w w^T with B block diagonal over the pairs (W, E)
// and (S, N).  Lane q forms the 2x2 block of its pair (p0, p1) = (q & 2, q | 1)
// exactly as its partner does, and row q of z = B^-1 w; a butterfly gives
// s = w.z.  apply() then takes a right-hand side (row rq on lane q, pressure
// entry r4), forms row q of y = B^-1 r, t = w.y by a butterfly, and returns
// row q of the solution with the pressure in pr.  Rows of wall edges are
// identity rows with rq = 0.
template <typename T>
struct TeamSolve {
  T B00, B01, B10, B11, idet, z, g, ga, iden, v3, ih;
  bool odd;
  // with_p = false: the 4x4 velocity block alone (the projection method's
  // intermediate-velocity block), solved as solve_vanka<T, 4> does
  template <class LV>
  __device__ __forceinline__ TeamSolve(const LV& L, int q, T dq, bool ap0, bool ap1, T b01, T b10,
                                       T vc, T A44, bool with_p = true) {
    ih = L.ih;
    v3 = vc * L.k.v3;
    odd = q & 1;
    T dqo = shfl_xor(dq, 1);
    T D0 = odd ? dqo : dq, D1 = odd ? dq : dqo;
    B00 = ap0 ? D0 - v3 : T(1);
    B11 = ap1 ? D1 - v3 : T(1);
    B01 = (ap0 && ap1) ? b01 : T(0);
    B10 = (ap0 && ap1) ? b10 : T(0);
    idet = qrcp(B00 * B11 - B01 * B10);
    T zn = odd ? ((ap1 ? B00 : T(0)) + (ap0 ? B10 : T(0))) : ((ap0 ? B11 : T(0)) + (ap1 ? B01 : T(0)));
    z = (odd ? -zn : zn) * idet;
    T sdot = odd ? -z : z;
    sdot += shfl_xor(sdot, 1);
    sdot += shfl_xor(sdot, 2);
    g = qrcp(T(1) + v3 * sdot);
    iden = with_p ? qrcp(A44 + L.k.ihaM * (sdot * g)) : T(0);
    ga = with_p ? g * L.k.ihM : T(0);
  }
  __device__ __forceinline__ T apply(T rq, T r4, T& pr) const {
    T rqo = shfl_xor(rq, 1);
    T r0 = odd ? rqo : rq, r1 = odd ? rq : rqo;
    T y = ((odd ? B00 : B11) * (odd ? r1 : r0) - (odd ? B10 : B01) * (odd ? r0 : r1)) * idet;
    T tdot = odd ? -y : y;
    tdot += shfl_xor(tdot, 1);
    tdot += shfl_xor(tdot, 2);
    const T tg = tdot * g;
    pr = (r4 + ih * tg) * iden;
    return y - z * (v3 * tg + ga * pr);
  }
  // the same for the transposed system: B transposed, the pressure column
  // -w/h, the pressure row a w (a = 1/(M h)); ap0, ap1 as in the constructor.
  // Sherman-Morrison's g and the pivot of p are the system's own.
  __device__ __forceinline__ T apply_t(T rq, T r4, bool ap0, bool ap1, T a, T& pr) const {
    T rqo = shfl_xor(rq, 1);
    T r0 = odd ? rqo : rq, r1 = odd ? rq : rqo;
    T y = ((odd ? B00 : B11) * (odd ? r1 : r0) - (odd ? B01 : B10) * (odd ? r0 : r1)) * idet;
    T zn = odd ? ((ap1 ? B00 : T(0)) + (ap0 ? B01 : T(0))) : ((ap0 ? B11 : T(0)) + (ap1 ? B10 : T(0)));
    T zt = (odd ? -zn : zn) * idet;
    T tdot = odd ? -y : y;
    tdot += shfl_xor(tdot, 1);
    tdot += shfl_xor(tdot, 2);
    const T tg = tdot * g;
    pr = (r4 - a * tg) * iden;
    return y - zt * (v3 * tg - ih * g * pr);
  }
};

// Vanka block of cell (i,j) by a team of four lanes (lane & 3 = q): lane q
// builds row q (diagonal entry and residual of edge q: W, E, S, N) and face
// q's share of the mass row; the team solves the 5x5 system together
// (TeamSolve); lane q writes edge q and lane 0 the pressure.  All 32 lanes of
// the warp call this (ok = false: a spare team, which computes on cell (1,1)
// and stores nothing).
template <typename T, class Form, class LV>
__device__ __forceinline__ void vanka_team(const Prm<T>& P, const LV& L, int i, int j, bool ok,
                                           T omega) {
  const int W = L.pitch;
  const int q = threadIdx.x & 3, d = q >> 1;
  const T ih = L.ih;
  int k = L.at(i, j);
  int eW = (L.px && i == 1) ? L.m1 : i - 1;
  int kW = L.at(eW, j);
  bool a0 = L.px || i > 1, a1 = L.px || i < L.m1, a2 = j > 1, a3 = j < L.m2;
  bool mine = q == 0 ? a0 : q == 1 ? a1 : q == 2 ? a2 : a3;
  int ke = q == 0 ? kW : (q == 2 ? k - W : k);
  // the neighbour across the edge's face; a periodic ghost holds the cell's copy
  const int nq = k + (q == 0 ? -1 : q == 1 ? 1 : q == 2 ? -W : W);
  const RhoPair<T> ra = rho_pair<T, Form>(P, L, k), rb = rho_pair<T, Form>(P, L, nq);
  const int kf = (q & 1) ? k : nq;  // the face's own edge (kW's copy for a periodic west face)
  T dq, bq;
  team_row<T, Form>(P, L, i, j, d, kf, ke, (q & 1) ? ra : rb, (q & 1) ? rb : ra, mine, dq, bq);
  // the mass row by faces: lane q takes face q (W, E, S, N) of the cell, the
  // face of its own edge: its velocity in d.u, its flux of
  // grad.(A m grad(mu + alpha p)) and, if open, its share of sum A m
  auto mob = L.mobn;
  T am = mob[nq] + mob[k];
  T f0 = team_sum<T>((q & 1) ? L.pair(d, L.u, L.v)[kf] : -L.pair(d, L.u, L.v)[kf]);
  T f1 = team_sum<T>(am * ((L.mu[nq] - L.mu[k]) + P.alpha * (L.p[nq] - L.p[k])));
  T f2 = team_sum<T>(mine ? am : T(0));
  T A44 = L.k.a2dif * f2;
  T b4 = f0 * ih - L.k.adif * f1 - L.fp[k];
  const T vc = L.visn[k];
  T b01, b10;
  pair_couplings<T, Form>(L, d, k, vc, b01, b10);
  TeamSolve<T> ts(L, q, dq, d ? a2 : a0, d ? a3 : a1, b01, b10, vc, A44);
  T pr;
  T x = ts.apply(bq, b4, pr);
  if (!ok) return;
  const bool ghosts = has_ghosts(L, i, j);
  const T xn = L.pair(d, L.u, L.v)[ke] - omega * x, pn = L.p[k] - omega * pr;
  if (mine) put_edge(L, i, j, q, ghosts, xn);
  if (q == 0) put_cell(L, L.p, i, j, ghosts, pn);
}

// One half of mom_residual for a lane pair of an eight-lane team: half 0 the
// time term (with gravity), the convection and -f; half 1 the pressure gradient,
// the surface tension and the viscous terms.  The two halves sum to the
// momentum row's N - f (up to the order of the additions).  FullForm only.
template <typename T, class LV>
__device__ __forceinline__ T mom_residual_half(const Prm<T>& P, const LV& L, int d, int k, T rl,
                                               T rr, int half) {
  const int s = d ? L.pitch : 1, t = d ? 1 : L.pitch;
  auto a = L.pair(d, L.u, L.v);
  auto b = L.pair(1 - d, L.u, L.v);
  T ae = a[k];
  T dl = (ae - a[k - s]) * L.ih, dr = (a[k + s] - ae) * L.ih;
  T Dp = (a[k + t] - ae) * L.ih, Dm = (ae - a[k - t]) * L.ih;
  if (half == 0) {
    auto S = L.pair(d, L.Sx, L.Sy);
    auto Q = L.pair(d, L.Qx, L.Qy);
    T conv = T(0.5) * (S[k + s] * dr + S[k] * dl + Q[k] * Dp + Q[k - t] * Dm);
    T time = ae * (L.pair(d, L.T1u, L.T1v)[k] + L.k.qidt * (rl + rr)) +
             L.pair(d, L.T0u, L.T0v)[k];
    return time + conv - L.pair(d, L.fu, L.fv)[k];
  }
  auto vis = L.visn;
  auto rn = L.rhon;
  T dvl = dl + (b[k] - b[k - t]) * L.ih;
  T dvr = dr + (b[k + s] - b[k + s - t]) * L.ih;
  T press = (L.p[k + s] - L.p[k]) * L.k.ihM;
  T st = -(rn[k + s] * L.mu[k] + rn[k] * L.mu[k + s]) * L.pair(d, L.Tx, L.Ty)[k] * P.iM;
  T vl = vis[k], vr = vis[k + s];
  T visc = -P.iRe * L.ih * ((vr * dr - vl * dl) + (L.Av[k] * Dp - L.Av[k - t] * Dm) +
                            (vr * dvr - vl * dvl) * T(1.0 / 3.0));
  return press + st + visc;
}

// Vanka block of cell (i,j) by a team of eight lanes (FP64 full iterate): as
// vanka_team, with each momentum row's residual split over the lane pair
// (q, q + 4) (mom_residual_half) and summed by one shuffle, so that each lane
// evaluates half a row.  Both halves of the team then run the same solve;
// the lower half stores.  For levels whose colour leaves most of the GPU idle:
// the visit's chain of dependent instructions is what bounds them.
template <typename T, class LV>
__device__ __forceinline__ void vanka_team8(const Prm<T>& P, const LV& L, int i, int j, bool ok,
                                            T omega) {
  const int W = L.pitch;
  const int q = threadIdx.x & 3, d = q >> 1, half = (threadIdx.x >> 2) & 1;
  const T ih = L.ih;
  int k = L.at(i, j);
  int eW = (L.px && i == 1) ? L.m1 : i - 1;
  int kW = L.at(eW, j);
  bool a0 = L.px || i > 1, a1 = L.px || i < L.m1, a2 = j > 1, a3 = j < L.m2;
  bool mine = q == 0 ? a0 : q == 1 ? a1 : q == 2 ? a2 : a3;
  int ke = q == 0 ? kW : (q == 2 ? k - W : k);
  T rl = L.rhoc[ke], rr = L.rhoc[ke + (d ? W : 1)];
  T dq = L.pair(d, L.Dgu, L.Dgv)[ke] + L.k.qidt * (rl + rr);
  T bq = mom_residual_half<T>(P, L, d, ke, rl, rr, half);
  bq += shfl_xor(bq, 4);
  if (!mine) bq = T(0);
  auto mob = L.mobn;
  const int nq = k + (q == 0 ? -1 : q == 1 ? 1 : q == 2 ? -W : W);
  T am = mob[nq] + mob[k];
  T f0 = team_sum<T>((q & 1) ? (d ? L.v[k] : L.u[k]) : -(d ? L.v[k - W] : L.u[k - 1]));
  T f1 = team_sum<T>(am * ((L.mu[nq] - L.mu[k]) + P.alpha * (L.p[nq] - L.p[k])));
  T f2 = team_sum<T>(mine ? am : T(0));
  T A44 = L.k.a2dif * f2;
  T b4 = f0 * ih - L.k.adif * f1 - L.fp[k];
  const T vc = L.visn[k];
  T b01, b10;
  pair_couplings<T, FullForm>(L, d, k, vc, b01, b10);
  TeamSolve<T> ts(L, q, dq, d ? a2 : a0, d ? a3 : a1, b01, b10, vc, A44);
  T pr;
  T x = ts.apply(bq, b4, pr);
  if (!ok || half) return;
  const bool ghosts = has_ghosts(L, i, j);
  const T xn = L.pair(d, L.u, L.v)[ke] - omega * x, pn = L.p[k] - omega * pr;
  if (mine) put_edge(L, i, j, q, ghosts, xn);
  if (q == 0) put_cell(L, L.p, i, j, ghosts, pn);
}

// The projection method's 4x4 intermediate-velocity block (vanka4_cell) by a
// team of four lanes: lane q builds row q (team_row without pressure, surface
// tension and gravity) and the team solves the block (TeamSolve without the
// pressure row); lane q writes edge q.
template <typename T, class LV>
__device__ __forceinline__ void vanka4_team(const Prm<T>& P, const LV& L, int i, int j, bool ok,
                                            T omega) {
  const int W = L.pitch;
  const int q = threadIdx.x & 3, d = q >> 1;
  int k = L.at(i, j);
  int eW = (L.px && i == 1) ? L.m1 : i - 1;
  int kW = L.at(eW, j);
  bool a0 = L.px || i > 1, a1 = L.px || i < L.m1, a2 = j > 1, a3 = j < L.m2;
  bool mine = q == 0 ? a0 : q == 1 ? a1 : q == 2 ? a2 : a3;
  int ke = q == 0 ? kW : (q == 2 ? k - W : k);
  // the neighbour across the edge's face; a periodic ghost holds the cell's copy
  const int nq = k + (q == 0 ? -1 : q == 1 ? 1 : q == 2 ? -W : W);
  const RhoPair<T> ra = rho_pair<T, ProjForm>(P, L, k), rb = rho_pair<T, ProjForm>(P, L, nq);
  const int kf = (q & 1) ? k : nq;  // the face's own edge (kW's copy for a periodic west face)
  T dq, bq;
  team_row<T, ProjForm>(P, L, i, j, d, kf, ke, (q & 1) ? ra : rb, (q & 1) ? rb : ra, mine, dq, bq);
  const T vc = L.visn[k];
  T b01, b10;
  pair_couplings<T, ProjForm>(L, d, k, vc, b01, b10);
  TeamSolve<T> ts(L, q, dq, d ? a2 : a0, d ? a3 : a1, b01, b10, vc, T(0), false);
  T pr;
  T x = ts.apply(bq, T(0), pr);
  if (!ok || !mine) return;
  put_edge(L, i, j, q, has_ghosts(L, i, j), L.pair(d, L.u, L.v)[ke] - omega * x);
}

// Coupled 7x7 block of coupled_cell by a team of four lanes (lane & 3 = q:
// edge and face W, E, S, N).  Lane q builds momentum row q, face q's terms of
// the mass row, of N_c, N_mu and of the CH Jacobian's face sums, and the
// couplings of edge q; butterflies add the face terms and every lane forms
// the cell terms.  The solve is solve_coupled7's by the NS block's structured
// solve (TeamSolve): the 2x2 Schur system for (dc, dmu), then the NS unknowns.
// Lane q writes edge q, lane 0 c, mu, p.
template <typename T, class Form, class LV>
__device__ __forceinline__ void coupled_team(const Prm<T>& P, const LV& L, int i, int j, bool ok,
                                             T omega) {
  const int W = L.pitch;
  const int q = threadIdx.x & 3, d = q >> 1;
  const T ih = L.ih;
  int k = L.at(i, j);
  int eW = (L.px && i == 1) ? L.m1 : i - 1;
  int kW = L.at(eW, j);
  bool a0 = L.px || i > 1, a1 = L.px || i < L.m1, a2 = j > 1, a3 = j < L.m2;
  bool mine = q == 0 ? a0 : q == 1 ? a1 : q == 2 ? a2 : a3;
  int ke = q == 0 ? kW : (q == 2 ? k - W : k);
  // the neighbour across the edge's face; a periodic ghost holds the cell's copy
  const int nq = k + (q == 0 ? -1 : q == 1 ? 1 : q == 2 ? -W : W);
  const RhoPair<T> ra = rho_pair<T, Form>(P, L, k), rb = rho_pair<T, Form>(P, L, nq);
  const int kf = (q & 1) ? k : nq;  // the face's own edge (kW's copy for a periodic west face)
  T dq, bq;
  team_row<T, Form>(P, L, i, j, d, kf, ke, (q & 1) ? ra : rb, (q & 1) ? rb : ra, mine, dq, bq);
  ChRows<T> C = ch_team_rows<T, Form>(P, L, i, j, q, mine, ra, rb);
  T sdiv = team_sum<T>((q & 1) ? L.pair(d, L.u, L.v)[kf] : -L.pair(d, L.u, L.v)[kf]);
  T sm = C.sm, sflux = C.sflux, gq = C.gq;
  T J11 = C.J11, J12 = C.J12, J21 = C.J21, J22 = C.J22, Rc = C.Rc, Rm = C.Rm;
  // the mass row and the couplings of edge q: d N_q/dc, d N_q/dmu (rows of
  // the two CH columns), d N_c/d x_q = g_q (the CH row), d N_p/dmu = d N_c/dp
  T A44 = L.k.a2dif * sm;
  T b4 = sdiv * ih - L.k.adif * sflux - L.fp[k];
  T diffc = L.k.adif * sm;
  T gm = mine ? gq : T(0);
  T cq0 = mine ? T(0.25) * C.drho * P.idt * (d ? Form::val_v(L, ke) : Form::val_u(L, ke)) : T(0);
  T cq1 = mine ? -gq * P.iM : T(0);
  const T vc = L.visn[k];
  T b01, b10;
  pair_couplings<T, Form>(L, d, k, vc, b01, b10);
  TeamSolve<T> ts(L, q, dq, d ? a2 : a0, d ? a3 : a1, b01, b10, vc, A44);
  // The Schur system of (dc, dmu) needs the CH row's products with the solved
  // columns, g^T A_NS^-1 r for three r: one transposed solve gives g^T A_NS^-1,
  // and one solve with the whole right-hand side then the NS unknowns (FP64
  // instructions, which bound the visit: 53 where three solves took 63; 96x144
  // coupled, three steps 19.6 -> 19.3 ms)
  T gp;
  const T gx = ts.apply_t(gm, diffc, d ? a2 : a0, d ? a3 : a1, L.k.ihM, gp);
  T S00 = J11 - team_sum<T>(gx * cq0);
  T S01 = J12 - (team_sum<T>(gx * cq1) + diffc * gp);
  T rhs0 = Rc - (team_sum<T>(gx * bq) + b4 * gp);
  T id2 = qrcp(S00 * J22 - S01 * J21);
  T dc = (J22 * rhs0 - S01 * Rm) * id2;
  T dm = (S00 * Rm - J21 * rhs0) * id2;
  T pr;
  T x = ts.apply(bq - cq0 * dc - cq1 * dm, b4 - diffc * dm, pr);
  if (!ok) return;
  const bool ghosts = has_ghosts(L, i, j);
  const T xn = L.pair(d, L.u, L.v)[ke] - omega * x, pn = L.p[k] - omega * pr;
  const T cnew = L.c[k] - omega * dc, mnew = L.mu[k] - omega * dm;
  if (mine) put_edge(L, i, j, q, ghosts, xn);
  if (q == 0) {
    put_cell(L, L.c, i, j, ghosts, cnew);
    if constexpr (!std::is_same<Form, ErrForm>::value)
      put_cell(L, L.rhoc, i, j, ghosts, rho_of(P, cnew));
    put_cell(L, L.mu, i, j, ghosts, mnew);
    put_cell(L, L.p, i, j, ghosts, pn);
  }
}

// Per-level launch with four lanes per Vanka block (vanka_team): a level whose
// colour leaves most SM sub-partitions idle runs each block's critical path
// split over four lanes.  Whole warps past the last team return together, so
// every warp that calls vanka_team has all 32 lanes in it.
template <typename T>
__global__ void __launch_bounds__(SNT, 4) k_vanka4_team(Prm<T> P, Lv<T> L, int colour, T omega) {
  pdl_enter();
  ColourSlots cs = vanka_slots(L, colour);
  int t = blockIdx.x * SNT + threadIdx.x;
  if ((t & ~31) >= 4 * cs.n) return;  // warp-uniform
  int i = 1, j = 1;
  bool ok = (t >> 2) < cs.n && vanka_slot_cell(L, colour, cs, t >> 2, i, j);
  if (!ok) i = j = 1;
  vanka4_team<T>(P, L, i, j, ok, omega);
}

template <typename T, class Form>
__global__ void __launch_bounds__(SNT, 4) k_coupled_team(Prm<T> P, Lv<T> L, int colour, T omega) {
  pdl_enter();
  ColourSlots cs = vanka_slots(L, colour);
  int t = blockIdx.x * SNT + threadIdx.x;
  if ((t & ~31) >= 4 * cs.n) return;  // warp-uniform
  int i = 1, j = 1;
  bool ok = (t >> 2) < cs.n && vanka_slot_cell(L, colour, cs, t >> 2, i, j);
  if (!ok) i = j = 1;
  coupled_team<T, Form>(P, L, i, j, ok, omega);
}

// per-level launch with eight lanes per Vanka block (vanka_team8; FP64 full
// iterate)
template <typename T>
__global__ void __launch_bounds__(SNT, 4) k_vanka_team8(Prm<T> P, Lv<T> L, int colour,
                                                     T omega) {
  pdl_enter();
  ColourSlots cs = vanka_slots(L, colour);
  int t = blockIdx.x * SNT + threadIdx.x;
  if ((t & ~31) >= 8 * cs.n) return;  // warp-uniform
  int i = 1, j = 1;
  bool ok = (t >> 3) < cs.n && vanka_slot_cell(L, colour, cs, t >> 3, i, j);
  if (!ok) i = j = 1;
  vanka_team8<T>(P, L, i, j, ok, omega);
}

template <typename T, class Form>
__global__ void __launch_bounds__(SNT, 4) k_vanka_team(Prm<T> P, Lv<T> L, int colour, T omega) {
  pdl_enter();
  ColourSlots cs = vanka_slots(L, colour);
  int t = blockIdx.x * SNT + threadIdx.x;
  if ((t & ~31) >= 4 * cs.n) return;  // warp-uniform
  int i = 1, j = 1;
  bool ok = (t >> 2) < cs.n && vanka_slot_cell(L, colour, cs, t >> 2, i, j);
  if (!ok) i = j = 1;
  vanka_team<T, Form>(P, L, i, j, ok, omega);
}

// Vanka block of cell (i,j) by a lane pair (FP64 full iterate; lane & 1 = d):
// lane 0 holds the x pair of the block (rows W, E), lane 1 the y pair (S, N).
// Each lane builds its two momentum rows (team_row) and its two faces of the
// mass row; one shuffle adds the faces.  The structured solve of solve_vanka
// then runs with each lane factoring only its own pair's 2x2 block B: s = w.z
// and t = w.y are the sums of the two pairs' shares, one shuffle each, and
// g, p and the pressure pivot are formed on both lanes alike.  Every sum is
// associated as in the four-lane team ((W + E) + (S + N)), so the arithmetic
// is the team's.  Against one lane per visit this halves each lane's FP64
// instructions, which is what bounds a launch whose colour fills the GPU
// more than once: the busiest sub-partition issues three warps of half a
// visit instead of two warps of a whole one.
template <typename T, class Form, class LV>
__device__ __forceinline__ void vanka_pair(const Prm<T>& P, const LV& L, int i, int j, bool ok,
                                           T omega) {
  const int W = L.pitch;
  const int d = threadIdx.x & 1;
  const T ih = L.ih;
  int k = L.at(i, j);
  int eW = (L.px && i == 1) ? L.m1 : i - 1;
  int kW = L.at(eW, j);
  bool a0 = L.px || i > 1, a1 = L.px || i < L.m1, a2 = j > 1, a3 = j < L.m2;
  // this lane's edges: the low one (W or S) and the high one (E or N)
  bool ap0 = d ? a2 : a0, ap1 = d ? a3 : a1;
  int ke0 = d ? k - W : kW;
  T dq0, bq0, dq1, bq1;
  {
    const int o = d ? W : 1;
    const RhoPair<T> rl = rho_pair<T, Form>(P, L, k - o), rk = rho_pair<T, Form>(P, L, k),
                     rr = rho_pair<T, Form>(P, L, k + o);
    team_row<T, Form>(P, L, i, j, d, k - o, ke0, rl, rk, ap0, dq0, bq0);
    team_row<T, Form>(P, L, i, j, d, k, k, rk, rr, ap1, dq1, bq1);
  }
  // the mass row by faces (as vanka_team): faces W, E on lane 0, S, N on lane 1
  auto mob = L.mobn;
  const int off = d ? W : 1;
  const int n0 = k - off, n1 = k + off;
  T am0 = mob[n0] + mob[k], am1 = mob[n1] + mob[k];
  T fs0 = -(d ? L.v[k - W] : L.u[k - 1]) + (d ? L.v[k] : L.u[k]);
  T fs1 = am0 * ((L.mu[n0] - L.mu[k]) + P.alpha * (L.p[n0] - L.p[k])) +
          am1 * ((L.mu[n1] - L.mu[k]) + P.alpha * (L.p[n1] - L.p[k]));
  T fs2 = (ap0 ? am0 : T(0)) + (ap1 ? am1 : T(0));
  fs0 += shfl_xor(fs0, 1);
  fs1 += shfl_xor(fs1, 1);
  fs2 += shfl_xor(fs2, 1);
  T A44 = L.k.a2dif * fs2;
  T b4 = fs0 * ih - L.k.adif * fs1 - L.fp[k];
  // this pair's block B = A_vv - v3 w w^T (TeamSolve, both rows on one lane)
  T vc = L.visn[k];
  T S = d ? L.Sy[k] : L.Sx[k];
  T v3 = vc * L.k.v3, v1 = vc * L.k.v1, sc = L.k.hih * S;
  T B00 = ap0 ? dq0 - v3 : T(1);
  T B11 = ap1 ? dq1 - v3 : T(1);
  T B01 = (ap0 && ap1) ? sc - v1 : T(0);
  T B10 = (ap0 && ap1) ? -sc - v1 : T(0);
  T idet = qrcp(B00 * B11 - B01 * B10);
  T z0 = ((ap0 ? B11 : T(0)) + (ap1 ? B01 : T(0))) * idet;
  T z1 = -((ap1 ? B00 : T(0)) + (ap0 ? B10 : T(0))) * idet;
  T sdot = z0 + -z1;
  sdot += shfl_xor(sdot, 1);
  T g = qrcp(T(1) + v3 * sdot);
  T iden = qrcp(A44 + L.k.ihaM * (sdot * g));
  T y0 = (B11 * bq0 - B01 * bq1) * idet;
  T y1 = (B00 * bq1 - B10 * bq0) * idet;
  T tdot = y0 + -y1;
  tdot += shfl_xor(tdot, 1);
  T tg = tdot * g;
  T pr = (b4 + ih * tg) * iden;
  T f = v3 * tg + (g * L.k.ihM) * pr;
  T x0 = y0 - z0 * f, x1 = y1 - z1 * f;
  if (!ok) return;
  if (d == 0) {
    if (ap0) store_u(L, eW, j, L.u[kW] - omega * x0);
    if (ap1) store_u(L, i, j, L.u[k] - omega * x1);
    store_cell(L, L.p, i, j, L.p[k] - omega * pr);
  } else {
    if (ap0) store_v(L, i, j - 1, L.v[k - W] - omega * x0);
    if (ap1) store_v(L, i, j, L.v[k] - omega * x1);
  }
}

// per-level launch with a lane pair per Vanka block (vanka_pair; FP64 full
// iterate).  Whole warps past the last pair return together.
template <typename T, class Form>
__global__ void __launch_bounds__(SNT, 4) k_vanka_pair(Prm<T> P, Lv<T> L, int colour, T omega) {
  pdl_enter();
  ColourSlots cs = vanka_slots(L, colour);
  int t = blockIdx.x * SNT + threadIdx.x;
  if ((t & ~31) >= 2 * cs.n) return;  // warp-uniform
  int i = 1, j = 1;
  bool ok = (t >> 1) < cs.n && vanka_slot_cell(L, colour, cs, t >> 1, i, j);
  if (!ok) i = j = 1;
  vanka_pair<T, Form>(P, L, i, j, ok, omega);
}

// per-level launch that splits a colour between one lane per block and lane
// pairs: slots [0, nsingle) one lane each (vanka_cell), the rest a lane pair
// each (vanka_pair), the single-lane warps first.  nsingle is a multiple of
// 32, so both branches are warp-uniform.  For a colour that fills the GPU's
// sub-partitions once and a fraction more (the finest level of the 256x512
// droplet: 820 warps on 608), a full round of single-lane warps followed by a
// round of pair warps for the remainder issues fewer FP64 instructions on the
// busiest sub-partition than a second, mostly empty single-lane round.
template <typename T, class Form>
__global__ void __launch_bounds__(SNT, 4) k_vanka_split(Prm<T> P, Lv<T> L, int colour, T omega,
                                                     int nsingle) {
  pdl_enter();
  ColourSlots cs = vanka_slots(L, colour);
  int t = blockIdx.x * SNT + threadIdx.x;
  if (t < nsingle) {
    int i, j;
    if (t < cs.n && vanka_slot_cell(L, colour, cs, t, i, j)) vanka_cell<T, Form>(P, L, i, j, omega);
    return;
  }
  int u = t - nsingle;
  if ((u & ~31) >= 2 * (cs.n - nsingle)) return;  // warp-uniform
  int sl = nsingle + (u >> 1), i = 1, j = 1;
  bool ok = sl < cs.n && vanka_slot_cell(L, colour, cs, sl, i, j);
  if (!ok) i = j = 1;
  vanka_pair<T, Form>(P, L, i, j, ok, omega);
}

// teams of four lanes while the colour fits in four warps per block of the
// fused group (one warp per sub-partition)
constexpr int QN_TEAM_MAX_SLOTS = 32;

template <typename T, class Form, class LV>
__device__ __forceinline__ void smooth_block(const Prm<T>& P, const LV& L, T omega, int coupled,
                                             int team8) {
  const int kcol = L.kcol;
  if constexpr (std::is_same<Form, ProjForm>::value) {
    // projection method (Sec. 7.2): CH red-black, intermediate-velocity blocks
    // over the Vanka colours, pressure Gauss-Seidel red-black
    const int mpr = L.crow.d;
    // four lanes per cell while a colour fits the block in one pass
    const bool cteam = 4 * mpr * L.m2 <= grp_size();
    for (int col = 0; col < 2; ++col) {
      if (cteam) {
        int t = grp_rank(), i = 1, j = 1;
        bool ok = (t >> 2) < mpr * L.m2 && ch_slot_cell(L, col, t >> 2, i, j);
        if (!ok) i = j = 1;
        if ((t & ~31) < 4 * mpr * L.m2) ch_team<T, Form>(P, L, i, j, ok);  // warp-uniform
      } else {
        for (int t = grp_rank(); t < mpr * L.m2; t += grp_size()) {
          int i, j;
          if (ch_slot_cell(L, col, t, i, j)) ch_cell<T, Form>(P, L, i, j);
        }
      }
      grp_sync();
    }
    for (int col = 0; col < kcol; ++col) {
      ColourSlots cs = vanka_slots(L, col);
      if (sizeof(T) == 8 && cs.n <= QN_TEAM_MAX_SLOTS * (int)gridDim.x) {  // one warp per sub-partition
        int t = grp_rank();
        if ((t & ~31) < 4 * cs.n) {  // warp-uniform: the warp holds at least one team
          int i = 1, j = 1;
          bool ok = (t >> 2) < cs.n && vanka_slot_cell(L, col, cs, t >> 2, i, j);
          if (!ok) i = j = 1;
          vanka4_team<T>(P, L, i, j, ok, omega);
        }
      } else {
        for (int t = grp_rank(); t < cs.n; t += grp_size()) {
          int i, j;
          if (vanka_slot_cell(L, col, cs, t, i, j)) vanka4_cell<T, Form>(P, L, i, j, omega);
        }
      }
      grp_sync();
    }
    for (int col = 0; col < 2; ++col) {
      if (cteam) {
        int t = grp_rank(), i = 1, j = 1;
        bool ok = (t >> 2) < mpr * L.m2 && ch_slot_cell(L, col, t >> 2, i, j);
        if (!ok) i = j = 1;
        if ((t & ~31) < 4 * mpr * L.m2) pgs_team<T>(P, L, i, j, ok);  // warp-uniform
      } else {
        for (int t = grp_rank(); t < mpr * L.m2; t += grp_size()) {
          int i, j;
          if (ch_slot_cell(L, col, t, i, j)) pgs_cell<T>(P, L, i, j);
        }
      }
      grp_sync();
    }
  } else {  // primitive method (full iterate or error equation)
  if (coupled) {
    for (int col = 0; col < kcol; ++col) {
      ColourSlots cs = vanka_slots(L, col);
      // four lanes per block while the colour fits the block in one pass
      if (lane_teams<T> && 4 * cs.n <= grp_size()) {
        int t = grp_rank();
        if ((t & ~31) < 4 * cs.n) {  // warp-uniform: the warp holds at least one team
          int i = 1, j = 1;
          bool ok = (t >> 2) < cs.n && vanka_slot_cell(L, col, cs, t >> 2, i, j);
          if (!ok) i = j = 1;
          if constexpr (lane_teams<T>) coupled_team<T, Form>(P, L, i, j, ok, omega);
        }
      } else {
        for (int t = grp_rank(); t < cs.n; t += grp_size()) {
          int i, j;
          if (vanka_slot_cell(L, col, cs, t, i, j)) coupled_cell<T, Form>(P, L, i, j, omega);
        }
      }
      grp_sync();
    }
    return;
  }
  const int mpr = L.crow.d;
  constexpr bool team_ok = std::is_same<Form, FullForm>::value && sizeof(T) == 8;
  constexpr bool vteam_ok = lane_teams<T>;
  for (int col = 0; col < 2; ++col) {
    if (vteam_ok && 4 * mpr * L.m2 <= grp_size()) {
      int t = grp_rank();
      if ((t & ~31) < 4 * mpr * L.m2) {  // warp-uniform
        int i = 1, j = 1;
        bool ok = (t >> 2) < mpr * L.m2 && ch_slot_cell(L, col, t >> 2, i, j);
        if (!ok) i = j = 1;
        if constexpr (vteam_ok) ch_team<T, Form>(P, L, i, j, ok);
      }
    } else {
      for (int t = grp_rank(); t < mpr * L.m2; t += grp_size()) {
        int i, j;
        if (ch_slot_cell(L, col, t, i, j)) ch_cell<T, Form>(P, L, i, j);
      }
    }
    grp_sync();
  }
  for (int col = 0; col < kcol; ++col) {
    ColourSlots cs = vanka_slots(L, col);
    // while the colour fits one warp per sub-partition of the group (full
    // iterate), or the group in one pass (FP64 error levels)
    const int team_slots = team_ok ? QN_TEAM_MAX_SLOTS * (int)gridDim.x : grp_size() / 4;
    if (team_ok && team8 && 8 * cs.n <= grp_size()) {  // eight lanes per block
      int t = grp_rank();
      if ((t & ~31) < 8 * cs.n) {  // warp-uniform: the warp holds at least one team
        int i = 1, j = 1;
        bool ok = (t >> 3) < cs.n && vanka_slot_cell(L, col, cs, t >> 3, i, j);
        if (!ok) i = j = 1;
        if constexpr (team_ok && LV::all_arrays) vanka_team8<T>(P, L, i, j, ok, omega);
      }
    } else if (vteam_ok && cs.n <= team_slots) {
      int t = grp_rank();
      if ((t & ~31) < 4 * cs.n) {  // warp-uniform: the warp holds at least one team
        int i = 1, j = 1;
        bool ok = (t >> 2) < cs.n && vanka_slot_cell(L, col, cs, t >> 2, i, j);
        if (!ok) i = j = 1;
        if constexpr (vteam_ok) vanka_team<T, Form>(P, L, i, j, ok, omega);
      }
    } else {
      for (int t = grp_rank(); t < cs.n; t += grp_size()) {
        int i, j;
        if (vanka_slot_cell(L, col, cs, t, i, j)) vanka_cell<T, Form>(P, L, i, j, omega);
      }
    }
    grp_sync();
  }
  }  // primitive method
}

// The V-cycle on the levels get(0) .. get(n - 1) as one loop over its level
// visits (down, coarsest, up), so that the smoother's code, the longest of the
// kernel, appears once: the visits of a colour step are bound by instruction
// latency, fetch included.
template <typename T, class Form, class Get>
__device__ __forceinline__ void coarse_vcycle_body(const Prm<T>& P, const Get& get, int n, int base,
                                                   int nu1, int nu2, int nuc, T omega, int coupled,
                                                   int team8) {
  double dummy[10];
  if constexpr (std::is_same<Form, ErrForm>::value) {
    for (int l = 1; base && l < n; ++l) {
      const auto& F = get(l - 1);
      const auto& G = get(l);
      for (int t = grp_rank(); t < (G.m1 + 1) * (G.m2 + 1); t += grp_size())
        restrict_base_cell(P, F, G, t % (G.m1 + 1), t / (G.m1 + 1));
      grp_sync();
    }
  }
  for (int visit = 0; visit < 2 * n - 1; ++visit) {
    const bool down = visit < n - 1, up = visit >= n;
    const int l = up ? 2 * n - 2 - visit : visit;
    const auto& F = get(l);
    if (up) {  // the correction from the level below
      const auto& G = get(l + 1);
      for (int t = grp_rank(); t < F.m1 * F.m2; t += grp_size())
        prolong_cell(P, F, G, t % F.m1 + 1, t / F.m1 + 1);
      grp_sync();
    }
    const int sweeps = down ? nu1 : up ? nu2 : nuc;
    for (int s = 0; s < sweeps; ++s) smooth_block<T, Form>(P, F, omega, coupled, team8);
    if (down) {
      const auto& G = get(l + 1);
      for (int t = grp_rank(); t < F.m1 * F.m2; t += grp_size())
        residual_cell<T, 0, Form>(P, F, t % F.m1 + 1, t / F.m1 + 1, dummy, false);
      grp_sync();
      for (int t = grp_rank(); t < (G.m1 + 1) * (G.m2 + 1); t += grp_size())
        restrict_state_cell(P, F, G, t % (G.m1 + 1), t / (G.m1 + 1));
      for (int t = grp_rank(); t < G.m1 * G.m2; t += grp_size())
        restrict_res_cell(F, G, t % G.m1 + 1, t / G.m1 + 1);
      grp_sync();
      for (int t = grp_rank(); t < G.m1 * G.m2; t += grp_size())
        residual_cell<T, 1, Form>(P, G, t % G.m1 + 1, t / G.m1 + 1, dummy, false);
      grp_sync();
    }
  }
}

// level l of a CoarseLevels
template <typename T>
struct LevelsOf {
  const CoarseLevels<T>& C;
  __device__ __forceinline__ const Lv<T>& operator()(int l) const { return C.L[l]; }
};

template <typename T, class Form, int NT>
__global__ void __launch_bounds__(NT, 1) k_coarse_vcycle(Prm<T> P, CoarseLevels<T> C, int nu1, int nu2,
                                                      int nuc, T omega, int coupled,
                                                      int team8) {
  pdl_enter();
  coarse_vcycle_body<T, Form>(P, LevelsOf<T>{C}, C.n, C.base, nu1, nu2, nuc, omega, coupled, team8);
}

// --------------------------------------------------------------------------
// The fused V-cycle of the FP64 full-iterate levels on a shared-memory copy.
// Its colour steps are chains of dependent loads and FP64 instructions of one
// visit each; from shared memory the loads take tens of cycles instead of an
// L2 round trip.  The block copies every array of its levels (QN_LV_ARRAYS,
// the padded frame [-1, m1+1] x [-1, m2+1] that the device code reads and
// writes) into shared memory at the compact pitch m1 + 3, runs the V-cycle
// body unchanged on level descriptors that point into the copy, and writes
// back the arrays the V-cycle writes: the unknowns, sources, residuals and the
// kept restricted iterate (the first 20 arrays) and rho(c).  For eight-lane
// Vanka blocks (vanka_team8), which read arrays that the records of
// k_coarse_records leave out.
// --------------------------------------------------------------------------
constexpr int QN_LV_NARR = 59;     // arrays of QN_LV_ARRAYS
constexpr int QN_LV_WRITTEN = 20;  // arrays 0..19 are written; and rho(c):
constexpr int QN_LV_RHOC = 44;

struct CoarseSmem {
  int off[QN_MAX_FUSED_LEVELS];  // first element of level l's copy
  long long ng[QN_MAX_FUSED_LEVELS];  // elements per array in the global block
  int head;  // elements (doubles) before the first copy: the descriptors
};

// copy arrays [q0, q1) of one level between its global block (pitch pg, ng
// elements per array) and its compact copy (pitch cc, rr rows).  Thread t
// takes column t % cw (cw >= cc) of rows t / cw + k NT / cw.  IN: global to
// shared by asynchronous copies (cp.async, 8 bytes each, all of a thread's in
// flight at once; the caller waits for them with cp.async.wait_all); else
// shared to global by plain stores.
template <int NT, bool IN>
__device__ __forceinline__ void coarse_copy(double* __restrict__ g, int pg, long long ng,
                                            double* __restrict__ sh, int cc, int rr, int q0,
                                            int q1) {
  const int cw = cc <= 16 ? 16 : 32, tx = threadIdx.x % cw, rstep = NT / cw;
  if (tx >= cc) return;
  const int ns = cc * rr;
  for (int r = threadIdx.x / cw; r < rr; r += rstep) {
    double* __restrict__ gr = g + (long long)r * pg + tx;
    double* __restrict__ sr = sh + r * cc + tx;
#pragma unroll 8
    for (int q = q0; q < q1; ++q) {
      if (IN) {
        const unsigned sa = (unsigned)__cvta_generic_to_shared(sr + q * ns);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gr + q * ng)
                     : "memory");
      } else {
        gr[q * ng] = sr[q * ns];
      }
    }
  }
}

template <int NT>
__global__ void __launch_bounds__(NT, 1) k_coarse_vcycle_smem(Prm<rf64> P, CoarseLevels<rf64> C,
                                                           CoarseSmem M, int nu1, int nu2,
                                                           int nuc, rf64 omega, int coupled,
                                                           int team8) {
  extern __shared__ __align__(16) double qn_coarse_smem[];
  pdl_enter();
  CoarseLevels<rf64>* S = reinterpret_cast<CoarseLevels<rf64>*>(qn_coarse_smem);
  double* arr = qn_coarse_smem + M.head;
  const int n = C.n;
  for (int l = 0; l < n; ++l) {
    const Lv<rf64>& G = C.L[l];
    const int cc = G.m1 + 3, rr = G.m2 + 3;
    coarse_copy<NT, true>(&G.c->v - (G.pitch + 1), G.pitch, M.ng[l], arr + M.off[l], cc, rr, 0,
                          QN_LV_NARR);
  }
  if (threadIdx.x < n) {  // the descriptor of level l, its arrays in the copy
    const int l = threadIdx.x;
    Lv<rf64> X = C.L[l];
    const int cc = X.m1 + 3, ns = cc * (X.m2 + 3);
    rf64* o = reinterpret_cast<rf64*>(arr + M.off[l] + cc + 1);  // origin (0,0) of array 0
    int q = 0;
#define QN_REBASE(m) X.m = o + (q++) * ns;
    QN_LV_ARRAYS(QN_REBASE)
#undef QN_REBASE
    X.pitch = cc;
    X.nst = ns;
    S->L[l] = X;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  coarse_vcycle_body<rf64, FullForm>(P, LevelsOf<rf64>{*S}, n, 0, nu1, nu2, nuc, omega, coupled,
                                       team8);
  __syncthreads();
  for (int l = 0; l < n; ++l) {
    const Lv<rf64>& G = C.L[l];
    const int cc = G.m1 + 3, rr = G.m2 + 3;
    double* g = &G.c->v - (G.pitch + 1);
    coarse_copy<NT, false>(g, G.pitch, M.ng[l], arr + M.off[l], cc, rr, 0, QN_LV_WRITTEN);
    coarse_copy<NT, false>(g, G.pitch, M.ng[l], arr + M.off[l], cc, rr, QN_LV_RHOC, QN_LV_RHOC + 1);
  }
}

// --------------------------------------------------------------------------
// The fused V-cycle on interleaved shared-memory records.  What a colour step
// cost beside its arithmetic was the chain of address arithmetic (a 64-bit
// address for each of the ~60 array elements a visit reads) and L2 round
// trips.  The copy interleaves the arrays that the V-cycle touches: a cell's
// values sit together, so that a visit forms three addresses (its row and the
// rows beside it) and reads everything else at constant offsets from them.  An
// odd number of values a cell keeps lanes on cells any power of two (or 5)
// apart in different banks.  The operators are the grid kernels' own
// (templates over the level), in the type whose rounding the source fixes, so
// the results are those of the launch that reads global memory.
// Measured (GB300, ncu, caches warm), FP32 error levels: 16x32 .. 2x4 of the
// 256x512 drop 245 -> 84 us, 28x28 and 14x14 of a served 448x448 request (64
// coupled sweeps on the coarsest) 1504 -> 630 us.  FP64: 8x16 .. 2x4 of the drop
// 290 -> 250 us, a 128x256 projection step's group 796 -> 721 us, the 6x9
// coupled group of 96x144 1618 -> 1435 us (the FP64 figures event-timed against
// global memory).  What is left is the
// chain of one warp's visit, colour after colour: per instruction issued it
// waits 1.2 cycles for a result in FP32 and 7.7 in FP64 (0.2 for code).  Two
// warps that shared a coupled visit (CH block; NS block and solve, the longer
// chain) were slower, 23.8 -> 24.6 ms for two served steps.
// --------------------------------------------------------------------------
// array OFF of records of N values at b: element k as if it were a plain array
template <typename T, int OFF, int N>
struct Fld {
  T* b;
  __device__ __forceinline__ T& operator[](int k) const { return b[k * N + OFF]; }
  __device__ __forceinline__ explicit operator bool() const { return true; }  // it is there
};
// A level in records (the members and constants of Lv); pairs of directions are
// neighbours in the record.  From level L and its record of cell (0,0) at b.
#define QN_RECORD_INDEX(m) I_##m,
#define QN_RECORD_MEMBER(m) Fld<T, I_##m, N> m;
#define QN_RECORD_SET(m) m.b = b;
#define QN_RECORD_LEVEL(NAME, ARRAYS, RHO)                                                     \
  template <typename T>                                                                        \
  struct NAME {                                                                                \
    typedef T real;                                                                            \
    enum { ARRAYS(QN_RECORD_INDEX) COUNT, N = COUNT | 1 };                                     \
    static constexpr bool has_rho = RHO, all_arrays = false;                                   \
    LvK<T> k;                                                                                  \
    FastDiv vrow, crow, kdiv;                                                                  \
    int m1, m2, px, pitch, kcol, c8;                                                           \
    T h, ih, ih2;                                                                              \
    ARRAYS(QN_RECORD_MEMBER)                                                                   \
    __device__ __forceinline__ NAME(const Lv<T>& L, T* b)                                      \
        : k(L.k), vrow(L.vrow), crow(L.crow), kdiv(L.kdiv), m1(L.m1), m2(L.m2), px(L.px),      \
          pitch(L.m1 + 3), kcol(L.kcol), c8(L.c8), h(L.h), ih(L.ih), ih2(L.ih2) {              \
      ARRAYS(QN_RECORD_SET)                                                                    \
    }                                                                                          \
    __device__ __forceinline__ int at(int i, int j) const { return j * pitch + i; }            \
    __device__ __forceinline__ int uhi() const { return px ? m1 : m1 - 1; }                    \
    template <int OFF>                                                                         \
    __device__ __forceinline__ Fld<T, OFF, N> pair(int d, Fld<T, OFF, N> x,                    \
                                                   Fld<T, OFF + 1, N>) const {                 \
      return {x.b + d};                                                                        \
    }                                                                                          \
    template <int OFF>                                                                         \
    __device__ __forceinline__ Fld<T, OFF, N> row_pair(int d, Fld<T, OFF, N> x,                \
                                                       Fld<T, OFF + 1, N>) const {             \
      return {x.b + d};                                                                        \
    }                                                                                          \
  }
// the unknowns, right-hand sides, residuals, the kept iterate; c^n and its fields
#define QN_COMMON_ARRAYS(X)                                                                    \
  X(c) X(mu) X(p) X(u) X(v) X(fc) X(fmu) X(fp) X(fu) X(fv) X(rc) X(rmu) X(rp) X(ru) X(rv)      \
  X(sc) X(smu) X(sp) X(su) X(sv) X(cn) X(rhon) X(mobn) X(visn) X(Gn) X(Tx) X(Ty)
// error equation: the rows' coefficients and the base
#define QN_ERR_ARRAYS(X)                                                                       \
  QN_COMMON_ARRAYS(X) X(T1u) X(T1v) X(aPu) X(aPv) X(aMu) X(aMv) X(tPu) X(tPv) X(tMu) X(tMv)    \
  X(Bc) X(Bmu) X(Bu) X(Bv) X(Bdc) X(rB)
// full iterate: rho(c), the rows' stencils, their diagonals and couplings; the
// projection method's rows hold their flux coefficients instead
#define QN_FULL_ARRAYS(X)                                                                      \
  QN_COMMON_ARRAYS(X) X(T0u) X(T0v) X(Cu) X(Cv) X(aPu) X(aPv) X(aMu) X(aMv) X(tPu) X(tPv)      \
  X(tMu) X(tMv) X(M0u) X(M0v) X(M1u) X(M1v) X(Dgu) X(Dgv) X(Sx) X(Sy) X(rhoc)
#define QN_PROJ_ARRAYS(X)                                                                      \
  QN_COMMON_ARRAYS(X) X(T0u) X(T0v) X(T1u) X(T1v) X(Dgu) X(Dgv) X(Sx) X(Sy) X(Qx) X(Qy) X(Av)  \
  X(rhoc)
QN_RECORD_LEVEL(LvErr, QN_ERR_ARRAYS, false);
QN_RECORD_LEVEL(LvFull, QN_FULL_ARRAYS, true);
QN_RECORD_LEVEL(LvProj, QN_PROJ_ARRAYS, true);

template <class Form>
struct RecordOf {  // FullForm
  template <typename T> using level = LvFull<T>;
  static constexpr int values = LvFull<rf64>::N;
};
template <>
struct RecordOf<ProjForm> {
  template <typename T> using level = LvProj<T>;
  static constexpr int values = LvProj<rf64>::N;
};
template <>
struct RecordOf<ErrForm> {
  template <typename T> using level = LvErr<T>;
  static constexpr int values = LvErr<rf32>::N;
};

struct RecordPlan {
  int off[QN_MAX_FUSED_LEVELS];  // first value of level l's records
};

template <typename T, class Form>
struct RecordLevels {
  const CoarseLevels<T>& C;
  const RecordPlan& M;
  T* base;
  __device__ __forceinline__ typename RecordOf<Form>::template level<T> operator()(int l) const {
    typedef typename RecordOf<Form>::template level<T> R;
    const Lv<T>& L = C.L[l];
    return R(L, base + M.off[l] + (L.m1 + 4) * R::N);  // cell (0,0) of the frame from (-1,-1)
  }
};

// copies array m of a level's records in (asynchronously)
template <typename T>
__device__ __forceinline__ void record_in(T* to, const T* from) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(to);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(sa), "l"(from),
               "n"((int)sizeof(T))
               : "memory");
}

template <typename T, class Form, int NT>
__global__ void __launch_bounds__(NT, 1) k_coarse_records(Prm<T> P,
                                                          const __grid_constant__ CoarseLevels<T> C,
                                                          const __grid_constant__ RecordPlan M,
                                                          int nu1, int nu2, int nuc, T omega,
                                                          int coupled) {
  typedef typename RecordOf<Form>::template level<T> R;
  extern __shared__ __align__(16) char qn_records[];
  T* const base = reinterpret_cast<T*>(qn_records);
  pdl_enter();
  const int n = C.n;
  for (int l = 0; l < n; ++l) {  // the padded frame of every array, all copies in flight at once
    const Lv<T>& L = C.L[l];
    const int cc = L.m1 + 3, cells = cc * (L.m2 + 3);
    for (int t = threadIdx.x; t < cells; t += NT) {
      const int g = (t / cc - 1) * L.pitch + t % cc - 1;
      T* const r = base + M.off[l] + t * R::N;
#define QN_RECORD_IN(m) record_in(r + R::I_##m, L.m + g);
      if constexpr (std::is_same<Form, ErrForm>::value) {
        QN_ERR_ARRAYS(QN_RECORD_IN)
      } else if constexpr (std::is_same<Form, ProjForm>::value) {
        QN_PROJ_ARRAYS(QN_RECORD_IN)
      } else {
        QN_FULL_ARRAYS(QN_RECORD_IN)
      }
#undef QN_RECORD_IN
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  coarse_vcycle_body<T, Form>(P, RecordLevels<T, Form>{C, M, base}, n, C.base, nu1, nu2, nuc, omega,
                              coupled, 0);
  __syncthreads();
  // what the levels above read of the group: the iterate of its finest level
  const Lv<T>& L = C.L[0];
  const int cc = L.m1 + 3, cells = cc * (L.m2 + 3);
  for (int t = threadIdx.x; t < cells; t += NT) {
    const int g = (t / cc - 1) * L.pitch + t % cc - 1;
    const T* r = base + M.off[0] + t * R::N;
    L.c[g] = r[R::I_c];
    L.mu[g] = r[R::I_mu];
    L.p[g] = r[R::I_p];
    L.u[g] = r[R::I_u];
    L.v[g] = r[R::I_v];
    if constexpr (R::has_rho) L.rhoc[g] = r[R::I_rhoc];
  }
}

// --------------------------------------------------------------------------
// banded wavefront of smoothing passes (one launch for nu smoothing steps on a
// level).  A smoothing step is a sequence of passes: CH red, CH black, then the
// Vanka colours (or the coupled block's colours).  Every visit reads and
// writes rows within 2 of its own, so with bands of at least 4 rows pass k on
// band b depends only on pass k - 1 on bands b - 1, b, b + 1.  Tickets are
// handed out in the order of t = b + 2k (then k), a topological order: a
// block takes a ticket, waits until each neighbouring band has finished pass
// k - 1 (per-band counters of finished passes), runs the pass's visits on its
// band and publishes the band's new count.  Each visit sees exactly the
// values it sees when every pass is a launch over the whole level and runs the
// same device code in the same type (Fused), so the results are those of the
// per-colour launches with as many lanes a visit; what changes is that a band's arrays stay in L2 across its
// passes instead of every colour launch streaming the whole level.
// A ticket's dependencies hold earlier tickets, taken by blocks that are
// running or done, so the wavefront progresses whatever the number of
// resident blocks.  Waits are bounded: past `budget` SM cycles a wait sets
// *flag (the step then fails with QNSCH_ETIMEOUT) and every later wait
// returns at once.
// --------------------------------------------------------------------------
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// the visits of pass `pass` on rows r0..r1 (1-based, inclusive)
template <typename T, class Form, class LV>
__device__ __forceinline__ void wave_pass(const Prm<T>& P, const LV& L, const WavePlan& W,
                                          int pass, int r0, int r1, T omega) {
  const int per = W.coupled ? L.kcol : L.kcol + 2;
  const int q = pass % per;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (!W.coupled && q < 2) {  // CH colour q: packed as in k_ch
    const int mpr = L.crow.d;
    const int t_lo = (r0 - 1) * mpr, t_hi = r1 * mpr;
    if (lane_teams<T> && mpr * L.m2 <= W.ch_team_max) {
      for (int base = t_lo; base < t_hi; base += nt / 4) {
        if (base + ((tid & ~31) >> 2) >= t_hi) continue;  // warp-uniform
        int t = base + (tid >> 2), i = 1, j = 1;
        bool ok = t < t_hi && ch_slot_cell(L, q, t, i, j);
        if (!ok) i = j = 1;
        if constexpr (lane_teams<T>) ch_team<T, Form>(P, L, i, j, ok);
      }
    } else {
      for (int t = t_lo + tid; t < t_hi; t += nt) {
        int i, j;
        if (ch_slot_cell(L, q, t, i, j)) ch_cell<T, Form>(P, L, i, j);
      }
    }
    return;
  }
  const int col = W.coupled ? q : q - 2;
  ColourSlots cs = vanka_slots(L, col);
  // the slots whose row j0 + rstep * (t / mpr) lies in [r0, r1]
  if (r1 < cs.j0) return;
  const int qlo = r0 > cs.j0 ? (r0 - cs.j0 + cs.rstep - 1) / cs.rstep : 0;
  const int qhi = (r1 - cs.j0) / cs.rstep;
  const int t_lo = qlo * cs.mpr, t_hi = min((qhi + 1) * cs.mpr, cs.n);
  if (lane_teams<T> && cs.n <= W.vanka_team_max) {
    for (int base = t_lo; base < t_hi; base += nt / 4) {
      if (base + ((tid & ~31) >> 2) >= t_hi) continue;  // warp-uniform
      int t = base + (tid >> 2), i = 1, j = 1;
      bool ok = t < t_hi && vanka_slot_cell(L, col, cs, t, i, j);
      if (!ok) i = j = 1;
      if constexpr (lane_teams<T>) {
        if (W.coupled) coupled_team<T, Form>(P, L, i, j, ok, omega);
        else vanka_team<T, Form>(P, L, i, j, ok, omega);
      }
    }
  } else {
    for (int t = t_lo + tid; t < t_hi; t += nt) {
      int i, j;
      if (!vanka_slot_cell(L, col, cs, t, i, j)) continue;
      if (W.coupled) coupled_cell<T, Form>(P, L, i, j, omega);
      else vanka_cell<T, Form>(P, L, i, j, omega);
    }
  }
}

constexpr int WAVE_NT = 256;

template <typename T, class Form>
__global__ void __launch_bounds__(WAVE_NT) k_wave(Prm<T> P, Lv<T> L, WavePlan W, T omega,
                                                  unsigned* ctr, double* flag) {
  pdl_enter();
  __shared__ unsigned s_t;
  unsigned* done = ctr + 1;
  const int N = W.nbands, K = W.npass;
  // tickets run over the (t = b + 2k, k) grid, t in [0, N + 2K - 2]
  const unsigned tickets = (unsigned)(N + 2 * K - 1) * (unsigned)K;
  for (;;) {
    if (threadIdx.x == 0) s_t = atomicAdd(ctr, 1u);
    __syncthreads();
    const unsigned t = s_t;
    __syncthreads();
    if (t >= tickets) break;
    const int tau = (int)(t / (unsigned)K), k = (int)(t % (unsigned)K), b = tau - 2 * k;
    if (b < 0 || b >= N) continue;  // a ticket of the grid with no band
    if (threadIdx.x == 0 && k > 0) {
      // pass k - 1 done on this band and its neighbours (test hook: one
      // wait for a count that nothing reaches)
      const unsigned need = (W.stall && b == 0 && k == 1) ? 0xffffffffu : (unsigned)k;
      const long long t0 = clock64();
      for (int nb = max(b - 1, 0); nb <= min(b + 1, N - 1); ++nb) {
        while (ld_acquire_u32(done + nb) < need) {
          if (*(volatile double*)flag != 0.0) break;
          if (clock64() - t0 > W.budget) {
            *(volatile double*)flag = 1.0;
            break;
          }
        }
      }
    }
    __syncthreads();
    const int r0 = b * W.rows + 1, r1 = min((b + 1) * W.rows, L.m2);
    wave_pass<T, Form>(P, L, W, k, r0, r1, omega);
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      st_release_u32(done + b, (unsigned)(k + 1));
    }
  }
}

// --------------------------------------------------------------------------
// skewed-chunk schedule of the smoothing passes on a large error-equation
// level.  A colour launch over the whole level touches every sector of every
// array its visits read (the visits of one colour are spread over all rows
// and columns), so a level larger than L2 streams from DRAM once per pass.
// Here the passes of a smoothing block run together over chunks of H rows:
// launch d runs pass p on the rows [1 + (d - p) H - 2p, 1 + (d - p + 1) H - 2p)
// (clipped to the level), so each pass trails the one before it by a chunk
// and two rows, and the rows the launch touches stay in L2 between the
// passes.  A visit at row j reads rows j - 2 .. j + 1 and writes rows j - 1
// and j (and the ghost row beside row 1 or row m2), so within one launch no
// task reads or writes what another task writes, every row a task reads
// already holds the results of the earlier passes (they ran in earlier
// launches) and none holds a later pass's: each visit sees the values it sees
// when every pass is a launch over the whole level, with the same device code.
// No block waits for another; stream order orders the launches.
// --------------------------------------------------------------------------
template <typename T, class Form, bool COUPLED>
__global__ void __launch_bounds__(SNT, 4) k_skew(Prm<T> P, Lv<T> L, SkewTasks S, T omega) {
  pdl_enter();
  const int b = blockIdx.x;
  int k = 0;
  while (k + 1 < S.n && S.boff[k + 1] <= b) ++k;
  const int t = S.t_lo[k] + (b - S.boff[k]) * SNT + threadIdx.x;
  if (t >= S.t_hi[k]) return;
  const int q = S.q[k];
  if constexpr (!COUPLED) {
    if (q < 2) {  // CH colour q, slots as in k_ch
      const int mpr = L.crow.d;
      int i, j;
      if (ch_slot_cell(L, q, t, i, j)) ch_cell<T, Form>(P, L, i, j);
      return;
    }
  }
  const int col = COUPLED ? q : q - 2;
  ColourSlots cs = vanka_slots(L, col);
  int i, j;
  if (!vanka_slot_cell(L, col, cs, t, i, j)) return;
  if constexpr (COUPLED) coupled_cell<T, Form>(P, L, i, j, omega);
  else vanka_cell<T, Form>(P, L, i, j, omega);
}

// --------------------------------------------------------------------------
// the predicted initial iterate of a step (option predictor): a Lagrange
// extrapolation in time of the committed state and the states before it,
// over the whole padded arrays (ghosts are linear in the values they copy,
// so the combination keeps them consistent)
// --------------------------------------------------------------------------
struct FiveArrays {
  double* p[5];
};

__global__ void __launch_bounds__(NT, 2) k_predict(FiveArrays X, FiveArrays A, FiveArrays B, FiveArrays C, double w0,
                          double w1, double w2, long long n, int off) {
  pdl_enter();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int q = blockIdx.y;
  const long long i = t - off;
  X.p[q][i] = w0 * A.p[q][i] + w1 * B.p[q][i] + w2 * C.p[q][i];
}

// --------------------------------------------------------------------------
// defect correction (mixed precision): FP64 level <-> error-equation level
// --------------------------------------------------------------------------
// These kernels move every array of a level once and are bound by its bytes.
// They read all of a cell's values before the first store: a load behind a
// store that may alias it waits for its turn, and a cell's ten loads in a row
// are ten round trips (k_start_correction on 1024x4096: 113 -> 91 us).
// error-equation frozen data = rounded FP64 frozen data (whole padded arrays)
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_cast_frozen(Lv<double> D, Lv<T> E, long long n, int off) {
  pdl_enter();
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  long long q = t - off;  // origin-relative index
  const double x[17] = {D.cn[q], D.rhon[q], D.mobn[q], D.visn[q], D.Gn[q], D.T1u[q], D.T1v[q],
                        D.aPu[q], D.aPv[q], D.aMu[q], D.aMv[q], D.tPu[q], D.tPv[q],
                        D.tMu[q], D.tMv[q], D.Tx[q], D.Ty[q]};
  T* const to[17] = {E.cn, E.rhon, E.mobn, E.visn, E.Gn, E.T1u, E.T1v, E.aPu, E.aPv, E.aMu,
                     E.aMv, E.tPu, E.tPv, E.tMu, E.tMv, E.Tx, E.Ty};
#pragma unroll
  for (int m = 0; m < 17; ++m) to[m][q] = (T)x[m];
}

// base X = x (rounded), X.c - c^n formed in FP64, right-hand side = FP64 residual
// (rounded), correction e = 0
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_start_correction(Prm<T> P, Lv<double> D, Lv<T> E, long long n, int off) {
  pdl_enter();
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  long long q = t - off;
  const double c = D.c[q], dc = c - D.cn[q], mu = D.mu[q], u = D.u[q], v = D.v[q];
  const double rc = D.rc[q], rmu = D.rmu[q], rp = D.rp[q], ru = D.ru[q], rv = D.rv[q];
  const T Bc = (T)c;
  E.Bc[q] = Bc;
  E.rB[q] = rho_of(P, Bc);
  E.Bmu[q] = (T)mu;
  E.Bu[q] = (T)u;
  E.Bv[q] = (T)v;
  E.Bdc[q] = (T)dc;
  E.fc[q] = (T)rc;
  E.fmu[q] = (T)rmu;
  E.fp[q] = (T)rp;
  E.fu[q] = (T)ru;
  E.fv[q] = (T)rv;
  E.c[q] = T(0);
  E.mu[q] = T(0);
  E.p[q] = T(0);
  E.u[q] = T(0);
  E.v[q] = T(0);
}

// x += e on the whole padded arrays (ghost rules are linear, so ghosts stay valid)
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_apply_correction(Prm<double> P, Lv<double> D, Lv<T> E, long long n, int off) {
  pdl_enter();
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  long long q = t - off;
  const double c = D.c[q] + (double)E.c[q], mu = D.mu[q] + (double)E.mu[q],
               p = D.p[q] + (double)E.p[q], u = D.u[q] + (double)E.u[q],
               v = D.v[q] + (double)E.v[q];
  D.c[q] = c;
  D.rhoc[q] = rho_of(P, c);
  D.mu[q] = mu;
  D.p[q] = p;
  D.u[q] = u;
  D.v[q] = v;
}

// rho(c) of the iterate over the whole padded array, after c was written in
// bulk (a new step's start, fields set from the host)
__global__ void __launch_bounds__(NT, 2) k_rho_fill(Prm<double> P, Lv<double> L, long long n, int off) {
  pdl_enter();
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  long long q = t - off;
  L.rhoc[q] = rho_of(P, L.c[q]);
}

// coarse base X_H = R X_h (cells: 4-mean; edges: 2 coincident fine edges)
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_restrict_base(Prm<T> P, Lv<T> F, Lv<T> C) {
  pdl_enter();
  int I = blockIdx.x * BX + threadIdx.x;
  int J = blockIdx.y * BY + threadIdx.y;
  if (I > C.m1 || J > C.m2) return;
  restrict_base_cell(P, F, C, I, J);
}

// --------------------------------------------------------------------------
// reductions
// --------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_sum_p(Lv<T> L, double* part) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x + 1;
  int j = blockIdx.y * BY + threadIdx.y + 1;
  double val[1] = {0.0};
  if (i <= L.m1 && j <= L.m2) val[0] = (double)L.p[L.at(i, j)];
  block_sum_store<1>(val, part, 0);
}

template <typename T>
__global__ void __launch_bounds__(NT, 2) k_sub_mean_p(Lv<T> L, const double* sum, double inv_n) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x;
  int j = blockIdx.y * BY + threadIdx.y;
  if (i > L.m1 + 1 || j > L.m2 + 1) return;
  L.p[L.at(i, j)] -= (T)(sum[0] * inv_n);
}

// mass: sum rho(c), sum rho(c) c over the cells (Thm. 6.1)
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_mass(Prm<T> P, Lv<T> L, const T* c, double* part) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x + 1;
  int j = blockIdx.y * BY + threadIdx.y + 1;
  double val[2] = {0.0, 0.0};
  if (i <= L.m1 && j <= L.m2) {
    double cc = (double)c[L.at(i, j)];
    double r = 1.0 / ((double)P.ia * cc + (double)P.ib);
    val[0] = r;
    val[1] = r * cc;
  }
  block_sum_store<2>(val, part, 0);
}

// --------------------------------------------------------------------------
// diagnostics of the experiments of Sec. 8 (FP64, committed state)
// --------------------------------------------------------------------------
// u_{i+1/2,j} for i = 0..m1 and v_{i,j+1/2} for j = 0..m2: zero on no-slip
// walls, period m1 in x
__device__ __forceinline__ double diag_u(const Lv<double>& L, const double* u, int i, int j) {
  if (!L.px && (i == 0 || i == L.m1)) return 0.0;
  if (L.px && i == 0) i = L.m1;
  return u[L.at(i, j)];
}
__device__ __forceinline__ double diag_v(const Lv<double>& L, const double* v, int i, int j) {
  if (j == 0 || j == L.m2) return 0.0;
  return v[L.at(i, j)];
}
// d_x u + d_y v of cell (i,j), by division: 1/h is itself rounded, which on a
// third of the sizes up to 1024 is up to 1.4 times the error
__device__ __forceinline__ double diag_div(const Lv<double>& L, const double* u, const double* v,
                                           int i, int j) {
  return (diag_u(L, u, i, j) - diag_u(L, u, i - 1, j)) / L.h +
         (diag_v(L, v, i, j) - diag_v(L, v, i, j - 1)) / L.h;
}

// per cell: [0] |div|, [1] max(div, 0), [2] max(-div, 0) (block maxima), then
// the sums [3] c, [4] c a_y(v), [5] c y, [6] div^2
__global__ void __launch_bounds__(NT, 2) k_diag_cells(Lv<double> L, const double* c, const double* u, const double* v,
                             double* part) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x + 1;
  int j = blockIdx.y * BY + threadIdx.y + 1;
  double val[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if (i <= L.m1 && j <= L.m2) {
    double d = diag_div(L, u, v, i, j);
    double cc = c[L.at(i, j)];
    double vbar = 0.5 * (diag_v(L, v, i, j) + diag_v(L, v, i, j - 1));
    val[0] = fabs(d);
    val[1] = fmax(d, 0.0);
    val[2] = fmax(-d, 0.0);
    val[3] = cc;
    val[4] = cc * vbar;
    val[5] = cc * ((j - 0.5) * L.h);
    val[6] = d * d;
  }
  block_sum_store<7>(val, part, 3);
}

// per cell: the upward crossing c_j >= 1/2 > c_{j+1} above it (linear between
// cell centres); [0] highest crossing, [1] Ly - lowest crossing (block maxima),
// then the sums [2] h c cos(2 pi x_i / Lx), whose column sums are eta_i = h
// sum_j c_ij, and [3] crossings.  A thread a cell: one thread a column walked
// its rows one load behind the other (row 1's block took 75 us on 256x512).
// The block's 32 cosines are formed once, by its first warp.
__global__ void __launch_bounds__(NT) k_diag_cols(Lv<double> L, const double* c, double* part) {
  pdl_enter();
  __shared__ double cosx[BX];
  const int i = blockIdx.x * BX + threadIdx.x + 1, j = blockIdx.y * BY + threadIdx.y + 1;
  const double h = L.h, Ly = L.m2 * h, Lx = L.m1 * h;
  if (threadIdx.y == 0) {
    const double pi = 3.14159265358979323846;
    cosx[threadIdx.x] = cos(2.0 * pi * ((i - 0.5) * h) / Lx);
  }
  __syncthreads();
  double val[4] = {0.0, 0.0, 0.0, 0.0};
  if (i <= L.m1 && j <= L.m2) {
    const double a = c[L.at(i, j)];
    val[2] = h * a * cosx[threadIdx.x];
    if (j < L.m2) {
      const double b = c[L.at(i, j + 1)];
      if (a >= 0.5 && b < 0.5) {
        const double y = (j - 0.5) * h + h * (a - 0.5) / (a - b);
        val[0] = y;
        val[1] = Ly - y;
        val[3] = 1.0;
      }
    }
  }
  block_sum_store<4>(val, part, 2);
}

// divergence field, packed out[(j-1)*m1 + (i-1)]
__global__ void k_div_field(Lv<double> L, const double* u, const double* v, double* out) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x + 1;
  int j = blockIdx.y * BY + threadIdx.y + 1;
  if (i > L.m1 || j > L.m2) return;
  out[(size_t)(j - 1) * L.m1 + (i - 1)] = diag_div(L, u, v, i, j);
}

// energy E_h (Thm. 6.2): per cell rho [a_x(u^2) + a_y(v^2)]/2 + (eps eta/(2We)) rho G(c)
// + (eta/(eps We)) rho F(c) + rho y / Fr; weights passed in w[0..2]
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_energy(Prm<T> P, Lv<T> L, const T* c, const T* u, const T* v, double w_grad,
                         double w_bulk, double w_pot, double* part) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x + 1;
  int j = blockIdx.y * BY + threadIdx.y + 1;
  double val[1] = {0.0};
  if (i <= L.m1 && j <= L.m2) {
    const int W = L.pitch;
    int k = L.at(i, j);
    double cc = (double)c[k];
    double r = 1.0 / ((double)P.ia * cc + (double)P.ib);
    double u0 = u[k], u1 = u[k - 1], v0 = v[k], v1 = v[k - W];
    double kin = 0.25 * (u0 * u0 + u1 * u1 + v0 * v0 + v1 * v1);
    double de = (double)c[k + 1] - cc, dw = cc - (double)c[k - 1];
    double dn = (double)c[k + W] - cc, ds = cc - (double)c[k - W];
    // (w_grad carries 1 / (2 h^2), w_bulk 1/4)
    double A = cc * (cc - 1.0);
    double y = (j - 0.5) * (double)L.h;
    val[0] = r * (kin + w_grad * (de * de + dw * dw + dn * dn + ds * ds) + w_bulk * (A * A) + w_pot * y);
  }
  block_sum_store<1>(val, part, 0);
}

// dissipation of Thm. 6.2 as sums of squares for the iterate against frozen data;
// thread (i,j) with i = 0..m1, j = 0..m2 handles vertex (i+1/2, j+1/2) and, for
// i, j >= 1, cell (i,j) and its east / north faces.  w: [dt/Re, dt/(3Re), dt/(M Pe)]
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_dissipation(Prm<T> P, Lv<T> L, double w_visc, double w_div, double w_ch,
                              double* part) {
  pdl_enter();
  int i = blockIdx.x * BX + threadIdx.x;
  int j = blockIdx.y * BY + threadIdx.y;
  double val[1] = {0.0};
  if (i <= L.m1 && j <= L.m2) {
    const int W = L.pitch;
    const double ih = 1.0 / (double)L.h;
    int k = L.at(i, j);
    double acc = 0.0;
    if (i >= 1 && j >= 1) {
      double rn = L.rhon[k], mv = L.visn[k];
      double du0 = (double)L.u[k] - L.un[k], du1 = (double)L.u[k - 1] - L.un[k - 1];
      double dv0 = (double)L.v[k] - L.vn[k], dv1 = (double)L.v[k - W] - L.vn[k - W];
      acc += 0.5 * rn * 0.5 * (du0 * du0 + du1 * du1 + dv0 * dv0 + dv1 * dv1);
      double dxu = ((double)L.u[k] - L.u[k - 1]) * ih, dyv = ((double)L.v[k] - L.v[k - W]) * ih;
      acc += w_visc * mv * (dxu * dxu + dyv * dyv) + w_div * mv * (dxu + dyv) * (dxu + dyv);
      double alpha = (double)P.alpha;
      double mc = (double)L.mu[k] + alpha * (double)L.p[k];
      if (L.px || i < L.m1) {
        double me = (double)L.mu[k + 1] + alpha * (double)L.p[k + 1];
        acc += w_ch * 0.5 * ((double)L.mobn[k] + L.mobn[k + 1]) * (me - mc) * (me - mc) * ih * ih;
      }
      if (j < L.m2) {
        double mn = (double)L.mu[k + W] + alpha * (double)L.p[k + W];
        acc += w_ch * 0.5 * ((double)L.mobn[k] + L.mobn[k + W]) * (mn - mc) * (mn - mc) * ih * ih;
      }
    }
    if (!L.px || i >= 1) {
      double Av = 0.25 * ((double)L.visn[k] + L.visn[k + 1] + L.visn[k + W] + L.visn[k + W + 1]);
      double Dyu = ((double)L.u[k + W] - L.u[k]) * ih;
      double Dxv = ((double)L.v[k + 1] - L.v[k]) * ih;
      double wy = (j == 0 || j == L.m2) ? 0.5 : 1.0;
      double wx = (!L.px && (i == 0 || i == L.m1)) ? 0.5 : 1.0;
      acc += w_visc * Av * (wy * Dyu * Dyu + wx * Dxv * Dxv);
    }
    val[0] = acc;
  }
  block_sum_store<1>(val, part, 0);
}

// --------------------------------------------------------------------------
// the outer-cycle loop of one step on the device (the step as one CUDA graph:
// a conditional WHILE node repeats the cycle, a conditional IF node commits).
// Control block ctl (doubles): [0] largest family residual r (scaled l2, NaN
// if any family is not finite), [1] cycles done k, [2] consecutive cycles the
// residual grew, [3] stopped by the time limit, [4] stopped by growth,
// [5] commit, [6..10] l2 norms, [11..15] max norms, [16] (as a 64-bit
// integer) the global timer in ns at the start of the step, [17] nonzero once
// a bounded wait of the wavefront smoother has run out.
// --------------------------------------------------------------------------
__device__ __forceinline__ long long global_ns() {
  long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__global__ void k_loop_clock(double* ctl) {
  pdl_enter();
  *reinterpret_cast<long long*>(ctl + 16) = global_ns();
}

// nrm: the norms of k_finalize ([0..4] max, [5..9] h^2 sum r^2).  The stopping
// rule is the host loop's: continue while r is finite, r > tol and k < maxcyc;
// stop after `diverge` consecutive cycles of growth; before a further cycle,
// stop as late once the step has run longer than limit_ns.
__global__ void k_loop_ctl(const double* nrm, double* ctl, cudaGraphConditionalHandle hl,
                           cudaGraphConditionalHandle hc, double tol, int maxcyc, int diverge,
                           double limit_ns, int first) {
  pdl_enter();
  double r = 0.0;
  bool nan = false;
  for (int q = 0; q < 5; ++q) {
    double l2 = sqrt(nrm[5 + q]);
    ctl[6 + q] = l2;
    ctl[11 + q] = nrm[q];
    if (!(l2 == l2)) nan = true;
    else if (l2 > r) r = l2;
  }
  if (nan) r = CUDART_NAN;
  double k = 0.0, grew = 0.0;
  if (!first) {
    k = ctl[1] + 1.0;
    grew = r > ctl[0] ? ctl[2] + 1.0 : 0.0;
  }
  const bool div = !first && diverge > 0 && grew >= (double)diverge;
  bool cont = !div && r == r && r > tol && k < (double)maxcyc;
  // a bounded wait of the wavefront smoother ran out (ctl[17] set): the cycle's
  // result is not to be trusted, the step ends as late
  bool late = ctl[17] != 0.0;
  if (late) cont = false;
  if (cont && limit_ns > 0.0 &&
      (double)(global_ns() - *reinterpret_cast<const long long*>(ctl + 16)) > limit_ns) {
    cont = false;
    late = true;
  }
  const bool commit = !cont && r == r && !late && r <= tol;
  ctl[0] = r;
  ctl[1] = k;
  ctl[2] = grew;
  ctl[3] = late ? 1.0 : 0.0;
  ctl[4] = div ? 1.0 : 0.0;
  ctl[5] = commit ? 1.0 : 0.0;
  cudaGraphSetConditional(hl, cont ? 1u : 0u);
  cudaGraphSetConditional(hc, commit ? 1u : 0u);
}

// --------------------------------------------------------------------------
// host layout <-> padded layout
// --------------------------------------------------------------------------
// kind 0: cell (m2 x m1), 1: u (m2 x (m1+1)), 2: v ((m2+1) x m1)
template <typename T>
__global__ void k_pack_in(Lv<T> L, T* dst, const double* src, int kind) {
  pdl_enter();
  int a = blockIdx.x * BX + threadIdx.x;
  int b = blockIdx.y * BY + threadIdx.y;
  int nx = kind == 1 ? L.m1 + 1 : L.m1, ny = kind == 2 ? L.m2 + 1 : L.m2;
  if (a >= nx || b >= ny) return;
  int I = kind == 1 ? a : a + 1, J = kind == 2 ? b : b + 1;
  dst[L.at(I, J)] = (T)src[(size_t)b * nx + a];
}
template <typename T>
__global__ void k_pack_out(Lv<T> L, double* dst, const T* src, int kind) {
  pdl_enter();
  int a = blockIdx.x * BX + threadIdx.x;
  int b = blockIdx.y * BY + threadIdx.y;
  int nx = kind == 1 ? L.m1 + 1 : L.m1, ny = kind == 2 ? L.m2 + 1 : L.m2;
  if (a >= nx || b >= ny) return;
  int I = kind == 1 ? a : a + 1, J = kind == 2 ? b : b + 1;
  dst[(size_t)b * nx + a] = (double)src[L.at(I, J)];
}

// ==========================================================================
// launchers
// ==========================================================================
static int frame_threads(int m1, int m2) { return 4 * (m1 + 3) + 4 * (m2 + 3); }

template <typename T>
int nparts_cells(const Lv<T>& L) {
  dim3 g = grid2(L.m1, L.m2);
  return g.x * g.y;
}

// Three threads a cell on FP64 full-iterate levels of at most 32768 cells: three
// threads' warps then still are at most five a sub-partition, and a launch is
// one thread's chain (a V-cycle of 256x256 2.16 -> 2.04 ms, a 64x64 step 7.72 ->
// 7.37 ms); on a level that fills the pipes the roles' shared loads and sums
// would be done three times.  (FP32 levels: a
// thread's chain is its loads, which the roles would repeat.)
template <typename T, class Form>
static bool residual_split(const Lv<compute_t<T, Form>>& L) {
  return !std::is_same<Form, ErrForm>::value && (long long)L.m1 * L.m2 <= 32768;
}
template <typename R, int MODE, class Form>
static void launch_residual_split(const Prm<R>& P, const Lv<R>& L, double* part, cudaStream_t s) {
  if constexpr (!std::is_same<Form, ErrForm>::value) {
    dim3 g = grid2(L.m1, L.m2);
    g.z = 3;
    qlaunch(&k_residual_split<R, MODE, Form>, g, dim3(BX, BY), 0, s, P, L, part);
  }
}
template <typename T, class Form>
void launch_residual(const Prm<T>& P0, const Lv<T>& L0, double* part, cudaStream_t s) {
  typedef compute_t<T, Form> R;
  const Prm<R>& P = as_compute<R>(P0);
  const Lv<R> L = as_compute<R>(level_consts(P0, L0));
  const int rows = residual_rows(L);
  if (rows == 8)
    qlaunch(&k_residual<R, 0, Form, 8>, grid2(L.m1, (L.m2 + 7) / 8), dim3(BX, BY), 0, s, P, L, part);
  else if (rows == 2)
    qlaunch(&k_residual<R, 0, Form, 2>, grid2(L.m1, (L.m2 + 1) / 2), dim3(BX, BY), 0, s, P, L, part);
  else if (residual_split<T, Form>(L))
    launch_residual_split<R, 0, Form>(P, L, part, s);
  else
    qlaunch(&k_residual<R, 0, Form, 1>, grid2(L.m1, L.m2), dim3(BX, BY), 0, s, P, L, part);
  ++g_launches;
}
template <typename T, class Form>
void launch_add_op(const Prm<T>& P0, const Lv<T>& L0, cudaStream_t s) {
  typedef compute_t<T, Form> R;
  const Prm<R>& P = as_compute<R>(P0);
  const Lv<R> L = as_compute<R>(level_consts(P0, L0));
  const int rows = residual_rows(L);
  if (rows == 8)
    qlaunch(&k_residual<R, 1, Form, 8>, grid2(L.m1, (L.m2 + 7) / 8), dim3(BX, BY), 0, s, P, L, nullptr);
  else if (rows == 2)
    qlaunch(&k_residual<R, 1, Form, 2>, grid2(L.m1, (L.m2 + 1) / 2), dim3(BX, BY), 0, s, P, L, nullptr);
  else if (residual_split<T, Form>(L))
    launch_residual_split<R, 1, Form>(P, L, nullptr, s);
  else
    qlaunch(&k_residual<R, 1, Form, 1>, grid2(L.m1, L.m2), dim3(BX, BY), 0, s, P, L, nullptr);
  ++g_launches;
}
template <typename T, class Form>
void launch_ch(const Prm<T>& P0, const Lv<T>& L0, int colour, cudaStream_t s, int team_max) {
  typedef compute_t<T, Form> R;
  const Prm<R>& P = as_compute<R>(P0);
  const Lv<R> L = as_compute<R>(level_consts(P0, L0));
  int n = (L.m1 + 1) / 2 * L.m2;
  if (n <= 0) return;
  if constexpr (lane_teams<T>) {
    if (n <= team_max) {  // four lanes per cell: shorter critical path per visit
      qlaunch(&k_ch_team<R, Form>, (4 * n + 63) / 64, 64, 0, s, P, L, colour);
      ++g_launches;
      return;
    }
  }
  qlaunch(&k_ch<R, Form>, (n + 63) / 64, 64, 0, s, P, L, colour);
  ++g_launches;
}
// SM sub-partitions of the current device (4 per SM)
static int sub_partitions() {
  static std::atomic<int> sms{0};
  if (!sms.load()) {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    sms = n > 0 ? n : 1;
  }
  return 4 * sms.load();
}

// Slots of an n-slot FP64 Vanka colour that k_vanka_split runs one lane per
// block (the rest run as lane pairs).  split >= 2 forces split rounded down to
// a multiple of 32; split == 1 picks the count by a cost model of the busiest
// sub-partition: ceil(warps / sub-partitions) rounds of single-lane warps cost
// one unit each, rounds of pair warps VANKA_PAIR_ROUND each (the measured
// ratio of a pair round to a single-lane round on the 256x512 droplet's finest
// level, 7.5 us against 10.4 us), for colours that need two rounds or more.
// Returns n when no split is cheaper.  The model's premise, that the rounds of
// a sub-partition add up, did not hold on that level: the split it picks
// (19,456 single-lane blocks, the rest in pairs) took 22.8 us against 20.7 us
// for one lane per block, whose time is set by one visit's chain per round.
constexpr double VANKA_PAIR_ROUND = 0.72;
int vanka_split_single(int n, int split) {
  if (split >= 2) return std::min(n, split / 32 * 32);
  const long long S = sub_partitions();
  const long long ws = (n + 31) / 32, rounds = (ws + S - 1) / S;
  // one round is bound by the latency of a visit's chain, which pairs do not shorten
  if (rounds < 2) return n;
  double best = (double)rounds;
  int ns = n;
  for (long long k = 0; k < rounds; ++k) {
    const long long single = std::min<long long>(n, k * S * 32);
    const long long pw = (2 * (n - single) + 31) / 32;
    const double cost = (double)k + VANKA_PAIR_ROUND * (double)((pw + S - 1) / S);
    if (cost < best) { best = cost; ns = (int)single; }
  }
  return ns;
}

template <typename T, class Form>
void launch_vanka(const Prm<T>& P0, const Lv<T>& L0, int colour, T omega, cudaStream_t s,
                  int team_max, int team8_max, int pair_max, int split) {
  typedef compute_t<T, Form> R;
  const Prm<R>& P = as_compute<R>(P0);
  const Lv<R> L = as_compute<R>(level_consts(P0, L0));
  int n = vanka_slots(L, colour).n;
  if (n <= 0) return;
  if constexpr (std::is_same<Form, FullForm>::value && sizeof(T) == 8) {
    if (n <= team8_max) {  // eight lanes per block: half a momentum row per lane
      qlaunch(&k_vanka_team8<R>, (8 * n + SNT - 1) / SNT, SNT, 0, s, P, L, colour, omega);
      ++g_launches;
      return;
    }
  }
  if constexpr (lane_teams<T>) {
    if (n <= team_max) {  // four lanes per block: shorter critical path per visit
      qlaunch(&k_vanka_team<R, Form>, (4 * n + SNT - 1) / SNT, SNT, 0, s, P, L, colour, omega);
      ++g_launches;
      return;
    }
  }
  if constexpr (std::is_same<Form, FullForm>::value && sizeof(T) == 8) {
    if (n <= pair_max) {  // a lane pair per block: half the FP64 instructions per lane
      qlaunch(&k_vanka_pair<R, Form>, (2 * n + SNT - 1) / SNT, SNT, 0, s, P, L, colour, omega);
      ++g_launches;
      return;
    }
    const int ns = split > 0 ? vanka_split_single(n, split) : n;
    if (ns < n) {  // one lane per block for slots [0, ns), a lane pair for the rest
      const long long threads = (long long)ns + 2LL * (n - ns);
      qlaunch(&k_vanka_split<R, Form>, (int)((threads + SNT - 1) / SNT), SNT, 0, s, P, L, colour,
              omega, ns);
      ++g_launches;
      return;
    }
  }
  qlaunch(&k_vanka<R, Form>, (n + SNT - 1) / SNT, SNT, 0, s, P, L, colour, omega);
  ++g_launches;
}
// shared memory a block of the current device may opt in to
static int smem_optin() {
  static std::atomic<int> optin{0};
  if (!optin.load()) {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    optin = v > 0 ? v : 1;
  }
  return optin.load();
}
// Plan of the shared-memory copy of an FP64 full-iterate fused group: every
// level's arrays at their block's stride in QN_LV_ARRAYS order (checked
// pointer by pointer), columns within the copy kernel's 32-wide rows, and the
// whole copy within the device's opt-in shared memory per block.  Returns the
// dynamic shared-memory bytes, 0 if the group does not qualify.
static size_t coarse_smem_plan(const Lv<double>* levels, int n, CoarseSmem& M) {
  const int head = (int)((sizeof(CoarseLevels<double>) + 15) / 16 * 2);
  long long elems = head;
  M.head = head;
  for (int l = 0; l < n; ++l) {
    const Lv<double>& L = levels[l];
    const int cc = L.m1 + 3, rr = L.m2 + 3;
    if (cc > 32 || !L.c) return 0;
    const long long ng = (long long)L.pitch * rr;
    int q = 0;
    bool ok = true;
#define QN_CHECK(m) ok = ok && L.m == L.c + (q++) * ng;
    QN_LV_ARRAYS(QN_CHECK)
#undef QN_CHECK
    if (!ok) return 0;
    M.ng[l] = ng;
    M.off[l] = (int)(elems - head);
    elems += (long long)QN_LV_NARR * cc * rr;
    elems = (elems + 1) / 2 * 2;  // 16-byte aligned copies
  }
  const size_t bytes = (size_t)elems * sizeof(double);
  return bytes <= (size_t)smem_optin() ? bytes : 0;
}

// Plan of k_coarse_records' copy; returns its bytes, 0 if it does not fit
template <typename T, class Form>
static size_t record_plan(const Lv<T>* levels, int n, RecordPlan& M) {
  const long long limit = smem_optin() / (long long)sizeof(T);
  long long values = 0;
  for (int l = 0; l < n; ++l) {
    M.off[l] = (int)values;
    values += (long long)(levels[l].m1 + 3) * (levels[l].m2 + 3) * RecordOf<Form>::values;
    if (values > limit) return 0;
  }
  return (size_t)values * sizeof(T);
}

void coarse_smem_prepare() {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
      v > 0) {
    cudaFuncSetAttribute(&k_coarse_vcycle_smem<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, v);
    cudaFuncSetAttribute(&k_coarse_records<rf32, ErrForm, 256>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, v);
    cudaFuncSetAttribute(&k_coarse_records<rf64, ErrForm, 256>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, v);
    cudaFuncSetAttribute(&k_coarse_records<rf64, FullForm, 256>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, v);
    cudaFuncSetAttribute(&k_coarse_records<rf64, ProjForm, 256>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, v);
  }
  cudaGetLastError();
}

template <typename T, class Form>
int launch_coarse_vcycle(const Prm<T>& P0, const Lv<T>* levels, int n, int nu1, int nu2, int nuc,
                         T omega, int coupled, cudaStream_t s, int team8, int ctas,
                         int smem) {
  typedef compute_t<T, Form> R;
  const Prm<R>& P = as_compute<R>(P0);
  CoarseLevels<R> C;
  C.n = n;
  C.base = std::is_same<Form, ErrForm>::value;
  for (int l = 0; l < n; ++l) C.L[l] = as_compute<R>(level_consts(P0, levels[l]));
  constexpr int NT = sizeof(T) == 8 ? 256 : 512;
  // eight lanes a block: the uncoupled FP64 primitive visits only (smooth_block)
  const bool eight = team8 && !coupled && std::is_same<Form, FullForm>::value && sizeof(T) == 8;
  if (smem && ctas <= 1 && !eight) {  // on shared-memory records, where they fit
    RecordPlan M = {};
    const size_t bytes = record_plan<T, Form>(levels, n, M);
    if (bytes) {
      qlaunch(&k_coarse_records<R, Form, 256>, 1, 256, bytes, s, P, C, M, nu1, nu2, nuc, R(omega),
              coupled);
      ++g_launches;
      return 1;
    }
  }
  if constexpr (std::is_same<Form, FullForm>::value && sizeof(T) == 8) {
    // eight-lane blocks read arrays that the records leave out: on a copy of all
    if (smem && ctas <= 1 && eight) {
      CoarseSmem M = {};
      const size_t bytes = coarse_smem_plan(levels, n, M);
      if (bytes) {
        qlaunch(&k_coarse_vcycle_smem<NT>, 1, NT, bytes, s, P, C, M, nu1, nu2, nuc, R(omega),
                coupled, team8);
        ++g_launches;
        return 1;
      }
    }
  }
  if (ctas <= 1) {
    qlaunch(&k_coarse_vcycle<R, Form, NT>, 1, NT, 0, s, P, C, nu1, nu2, nuc, omega, coupled,
            team8);
  } else {  // one cluster of ctas blocks (a size coarse_cluster_blocks accepted)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(NT);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g_pdl ? 2 : 1;
    cudaLaunchKernelEx(&cfg, &k_coarse_vcycle<R, Form, NT>, P, C, nu1, nu2, nuc, omega,
                       coupled, team8);
  }
  ++g_launches;
  return 0;
}

// largest cluster of at most `ctas` blocks (a power of two) in which the fused
// V-cycle of this form can run on the current device: a cluster is placed on
// the SMs of one GPC as a whole, and sizes above 8 need the non-portable
// cluster attribute, which the function must accept
template <typename T, class Form>
static int cluster_fit(int ctas) {
  constexpr int NT = sizeof(T) == 8 ? 256 : 512;
  auto kern = &k_coarse_vcycle<compute_t<T, Form>, Form, NT>;
  if (ctas > 8 &&
      cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    ctas = 8;
  }
  for (; ctas > 1; ctas >>= 1) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(NT);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) == cudaSuccess && nclusters > 0)
      break;
    cudaGetLastError();
  }
  return ctas < 1 ? 1 : ctas;
}

int coarse_cluster_blocks(int ctas) {
  int c = 1;
  while (c < 16 && 2 * c <= ctas) c *= 2;
  if (c == 1) return 1;
  c = cluster_fit<double, FullForm>(c);
  c = cluster_fit<double, ErrForm>(c);
  c = cluster_fit<float, ErrForm>(c);
  c = cluster_fit<double, ProjForm>(c);
  return c;
}

template <typename T, class Form>
void launch_vanka4(const Prm<T>& P0, const Lv<T>& L0, int colour, T omega, cudaStream_t s,
                   int team_max) {
  typedef compute_t<T, Form> R;
  const Prm<R>& P = as_compute<R>(P0);
  const Lv<R> L = as_compute<R>(level_consts(P0, L0));
  int n = vanka_slots(L, colour).n;
  if (n <= 0) return;
  if constexpr (std::is_same<Form, ProjForm>::value && sizeof(T) == 8) {
    if (n <= team_max) {  // four lanes per block: shorter critical path per visit
      qlaunch(&k_vanka4_team<R>, (4 * n + SNT - 1) / SNT, SNT, 0, s, P, L, colour, omega);
      ++g_launches;
      return;
    }
  }
  qlaunch(&k_vanka4<R, Form>, (n + SNT - 1) / SNT, SNT, 0, s, P, L, colour, omega);
  ++g_launches;
}
template <typename T>
void launch_pgs(const Prm<T>& P0, const Lv<T>& L0, int colour, cudaStream_t s, int team_max) {
  typedef compute_t<T, ProjForm> R;
  const Prm<R>& P = as_compute<R>(P0);
  const Lv<R> L = as_compute<R>(level_consts(P0, L0));
  int n = (L.m1 + 1) / 2 * L.m2;
  if (n <= 0) return;
  if (n <= team_max) {  // four lanes per cell: shorter critical path per visit
    qlaunch(&k_pgs_team<R>, (4 * n + 63) / 64, 64, 0, s, P, L, colour);
    ++g_launches;
    return;
  }
  qlaunch(&k_pgs<R>, (n + 63) / 64, 64, 0, s, P, L, colour);
  ++g_launches;
}
template <typename T>
void launch_proj_velocity(const Prm<T>& P, const Lv<T>& L0, T* uo, T* vo, cudaStream_t s) {
  const Lv<T> L = level_consts(P, L0);
  qlaunch(&k_proj_velocity<T>, grid2(L.m1 + 1, L.m2 + 1), dim3(BX, BY), 0, s, P, L, uo, vo);
  ++g_launches;
}
template <typename T>
void launch_proj_diss(const Prm<T>& P, const Lv<T>& L, const T* uo, const T* vo, double* part,
                      double* out1, cudaStream_t s) {
  qlaunch(&k_proj_diss<T>, grid2(L.m1, L.m2), dim3(BX, BY), 0, s, P, L, uo, vo, part);
  ++g_launches;
  qlaunch(&k_finalize, 1, FIN_NT, 0, s, part, nparts_cells(L), 1, 0, 0.5 * (double)L.h * (double)L.h, out1);
  ++g_launches;
}
template <typename T, class Form>
void launch_coupled(const Prm<T>& P0, const Lv<T>& L0, int colour, T omega, cudaStream_t s,
                    int team_max) {
  typedef compute_t<T, Form> R;
  const Prm<R>& P = as_compute<R>(P0);
  const Lv<R> L = as_compute<R>(level_consts(P0, L0));
  int n = vanka_slots(L, colour).n;
  if (n <= 0) return;
  if constexpr (lane_teams<T>) {
    if (n <= team_max) {  // four lanes per block: shorter critical path per visit
      qlaunch(&k_coupled_team<R, Form>, (4 * n + SNT - 1) / SNT, SNT, 0, s, P, L, colour, omega);
      ++g_launches;
      return;
    }
  }
  qlaunch(&k_coupled<R, Form>, (n + SNT - 1) / SNT, SNT, 0, s, P, L, colour, omega);
  ++g_launches;
}

static long long padded_n(int m1, int m2) {
  long long pitch = ((m1 + 3) + 31) / 32 * 32;
  return pitch * (m2 + 3);
}
template <typename T>
void launch_cast_frozen(const Lv<double>& D, const Lv<T>& E, cudaStream_t s) {
  long long n = padded_n(D.m1, D.m2);
  qlaunch(&k_cast_frozen<T>, (unsigned)((n + 255) / 256), 256, 0, s, D, E, n, D.pitch + 1);
  ++g_launches;
}
template <typename T>
void launch_start_correction(const Prm<T>& P, const Lv<double>& D, const Lv<T>& E, cudaStream_t s) {
  long long n = padded_n(D.m1, D.m2);
  qlaunch(&k_start_correction<T>, (unsigned)((n + 255) / 256), 256, 0, s, P, D, E, n, D.pitch + 1);
  ++g_launches;
}
template <typename T>
void launch_apply_correction(const Prm<double>& P, const Lv<double>& D, const Lv<T>& E,
                             cudaStream_t s) {
  long long n = padded_n(D.m1, D.m2);
  qlaunch(&k_apply_correction<T>, (unsigned)((n + 255) / 256), 256, 0, s, P, D, E, n, D.pitch + 1);
  ++g_launches;
}
void launch_rho_fill(const Prm<double>& P, const Lv<double>& L, cudaStream_t s) {
  long long n = padded_n(L.m1, L.m2);
  qlaunch(&k_rho_fill, (unsigned)((n + 255) / 256), 256, 0, s, P, L, n, L.pitch + 1);
  ++g_launches;
}
template <typename T>
void launch_restrict_base(const Prm<T>& P, const Lv<T>& F, const Lv<T>& C, cudaStream_t s) {
  qlaunch(&k_restrict_base<T>, grid2(C.m1 + 1, C.m2 + 1), dim3(BX, BY), 0, s, P, F, C);
  ++g_launches;
}
template <typename T>
void launch_bc_unknowns(const Lv<T>& L, cudaStream_t s) {
  int n = frame_threads(L.m1, L.m2);
  qlaunch(&k_bc_unknowns<T>, (n + 255) / 256, 256, 0, s, L);
  ++g_launches;
}
template <typename T>
void launch_frozen(const Prm<T>& P, const Lv<T>& L, cudaStream_t s) {
  int n = frame_threads(L.m1, L.m2);
  qlaunch(&k_bc_frozen<T>, (n + 255) / 256, 256, 0, s, L);
  ++g_launches;
  qlaunch(&k_frozen_derived<T>, grid2(L.m1 + 2, L.m2 + 2), dim3(BX, BY), 0, s, P, L);
  ++g_launches;
  qlaunch(&k_frozen_coef1<T>, grid2(L.m1 + 2, L.m2 + 2), dim3(BX, BY), 0, s, L);
  ++g_launches;
  qlaunch(&k_frozen_coef2<T>, grid2(L.m1 + 1, L.m2 + 1), dim3(BX, BY), 0, s, L);
  if (L.T1u) {  // FP64 full-iterate levels
    qlaunch(&k_frozen_coef3<T>, grid2(L.m1 + 1, L.m2 + 1), dim3(BX, BY), 0, s, P, L);
    ++g_launches;
  }
  ++g_launches;
}
template <typename T>
void launch_restrict(const Prm<T>& P, const Lv<T>& F, const Lv<T>& C, cudaStream_t s) {
  qlaunch(&k_restrict<T>, grid2(C.m1 + 1, C.m2 + 1), dim3(BX, BY), 0, s, P, F, C);
  ++g_launches;
}
template <typename T>
void launch_restrict_frozen(const Lv<T>& F, const Lv<T>& C, cudaStream_t s) {
  qlaunch(&k_restrict_frozen<T>, grid2(C.m1 + 1, C.m2 + 1), dim3(BX, BY), 0, s, F, C);
  ++g_launches;
}
template <typename T>
void launch_prolong(const Prm<T>& P, const Lv<T>& F, const Lv<T>& C, cudaStream_t s) {
  qlaunch(&k_prolong<T>, grid2(F.m1, F.m2), dim3(BX, BY), 0, s, P, F, C);
  ++g_launches;
}
template <typename T>
void launch_gauge(const Lv<T>& L, double* part, double* scal, cudaStream_t s) {
  qlaunch(&k_sum_p<T>, grid2(L.m1, L.m2), dim3(BX, BY), 0, s, L, part);
  ++g_launches;
  qlaunch(&k_finalize, 1, FIN_NT, 0, s, part, nparts_cells(L), 1, 0, 1.0, scal);
  ++g_launches;
  qlaunch(&k_sub_mean_p<T>, grid2(L.m1 + 2, L.m2 + 2), dim3(BX, BY), 0, s, L, scal,
                                                                     1.0 / ((double)L.m1 * L.m2));
  ++g_launches;
}
template <typename T>
void launch_norms_finalize(const Lv<T>& L, double* part, double* out10, cudaStream_t s) {
  // part rows are [max x5, sum of squares x5]; out10 = [l2 x5, max x5] after the
  // host applies sqrt(h^2 *) to the sums; here: out[0..4] = max, out[5..9] = h^2 sum
  dim3 g = grid2(L.m1, (L.m2 + residual_rows(L) - 1) / residual_rows(L));  // k_residual's blocks
  qlaunch(&k_finalize, 1, FIN_NT, 0, s, part, (int)(g.x * g.y), 10, 5, (double)L.h * (double)L.h, out10);
  ++g_launches;
}
void launch_diag(const Lv<double>& L, const double* c, const double* u, const double* v,
                 double* part, double* out11, cudaStream_t s) {
  qlaunch(&k_diag_cells, grid2(L.m1, L.m2), dim3(BX, BY), 0, s, L, c, u, v, part);
  qlaunch(&k_finalize, 1, FIN_NT, 0, s, part, nparts_cells(L), 7, 3, 1.0, out11);
  qlaunch(&k_diag_cols, grid2(L.m1, L.m2), dim3(BX, BY), 0, s, L, c, part);
  qlaunch(&k_finalize, 1, FIN_NT, 0, s, part, nparts_cells(L), 4, 2, 1.0, out11 + 7);
  g_launches += 4;
}
void launch_div_field(const Lv<double>& L, const double* u, const double* v, double* out,
                      cudaStream_t s) {
  qlaunch(&k_div_field, grid2(L.m1, L.m2), dim3(BX, BY), 0, s, L, u, v, out);
  ++g_launches;
}
template <typename T>
void launch_mass(const Prm<T>& P, const Lv<T>& L, const T* c, double* part, double* out2,
                 cudaStream_t s) {
  qlaunch(&k_mass<T>, grid2(L.m1, L.m2), dim3(BX, BY), 0, s, P, L, c, part);
  ++g_launches;
  qlaunch(&k_finalize, 1, FIN_NT, 0, s, part, nparts_cells(L), 2, 0, (double)L.h * (double)L.h, out2);
  ++g_launches;
}
template <typename T>
void launch_energy(const Prm<T>& P, const Lv<T>& L, const T* c, const T* u, const T* v,
                   double w_grad, double w_bulk, double w_pot, double* part, double* out1,
                   cudaStream_t s) {
  const double h = L.h;
  qlaunch(&k_energy<T>, grid2(L.m1, L.m2), dim3(BX, BY), 0, s, P, L, c, u, v, w_grad * 0.5 / (h * h),
          0.25 * w_bulk, w_pot, part);
  ++g_launches;
  qlaunch(&k_finalize, 1, FIN_NT, 0, s, part, nparts_cells(L), 1, 0, (double)L.h * (double)L.h, out1);
  ++g_launches;
}
template <typename T>
void launch_dissipation(const Prm<T>& P, const Lv<T>& L, double w_visc, double w_div,
                        double w_ch, double* part, double* out1, cudaStream_t s) {
  dim3 g = grid2(L.m1 + 1, L.m2 + 1);
  qlaunch(&k_dissipation<T>, g, dim3(BX, BY), 0, s, P, L, w_visc, w_div, w_ch, part);
  ++g_launches;
  qlaunch(&k_finalize, 1, FIN_NT, 0, s, part, g.x * g.y, 1, 0, (double)L.h * (double)L.h, out1);
  ++g_launches;
}
template <typename T>
void launch_pack_in(const Lv<T>& L, T* dst, const double* src, int kind, cudaStream_t s) {
  int nx = kind == 1 ? L.m1 + 1 : L.m1, ny = kind == 2 ? L.m2 + 1 : L.m2;
  qlaunch(&k_pack_in<T>, grid2(nx, ny), dim3(BX, BY), 0, s, L, dst, src, kind);
  ++g_launches;
}
template <typename T>
void launch_pack_out(const Lv<T>& L, double* dst, const T* src, int kind, cudaStream_t s) {
  int nx = kind == 1 ? L.m1 + 1 : L.m1, ny = kind == 2 ? L.m2 + 1 : L.m2;
  qlaunch(&k_pack_out<T>, grid2(nx, ny), dim3(BX, BY), 0, s, L, dst, src, kind);
  ++g_launches;
}

template <typename T, class Form>
void launch_wave(const Prm<T>& P0, const Lv<T>& L0, const WavePlan& W, T omega, unsigned* ctr,
                 double* flag, cudaStream_t s) {
  typedef compute_t<T, Form> R;
  const Prm<R>& P = as_compute<R>(P0);
  const Lv<R> L = as_compute<R>(level_consts(P0, L0));
  static std::atomic<int> blocks_per_sm{0};
  static std::atomic<int> sms{0};
  if (!sms.load()) {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    sms = n > 0 ? n : 1;
  }
  if (!blocks_per_sm.load()) {
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_wave<R, Form>, WAVE_NT, 0);
    blocks_per_sm = b > 0 ? b : 1;
  }
  const long long tasks = (long long)W.nbands * W.npass;
  const int grid = (int)std::min<long long>((long long)sms.load() * blocks_per_sm.load(), tasks);
  cudaMemsetAsync(ctr, 0, (size_t)(1 + W.nbands) * sizeof(unsigned), s);
  qlaunch(&k_wave<R, Form>, grid, WAVE_NT, 0, s, P, L, W, omega, ctr, flag);
  ++g_launches;
}

template <typename T, class Form>
int launch_skew(const Prm<T>& P0, const Lv<T>& L0, int nsteps, int coupled, int rows, T omega,
                cudaStream_t s) {
  typedef compute_t<T, Form> R;
  const Prm<R>& P = as_compute<R>(P0);
  const Lv<R> L = as_compute<R>(level_consts(P0, L0));
  const int per = coupled ? L.kcol : L.kcol + 2;
  const int H = std::max(rows, 1);
  const int group = std::max(1, SKEW_MAX_TASKS / per);  // steps per schedule
  int launches = 0;
  for (int s0 = 0; s0 < nsteps; s0 += group) {
    const int npass = std::min(group, nsteps - s0) * per;
    // the last diagonal on which the last pass still has rows of the level
    const int D = npass + (L.m2 - 1 + (npass - 1) * SKEW_LAG) / H;
    for (int d = 0; d < D; ++d) {
      SkewTasks S;
      S.n = 0;
      int nb = 0;
      for (int p = 0; p < npass; ++p) {
        const int lo = std::max(1 + (d - p) * H - p * SKEW_LAG, 1);
        const int hi = std::min(1 + (d - p + 1) * H - p * SKEW_LAG, L.m2 + 1);
        if (lo >= hi) continue;
        const int q = p % per;
        int t_lo, t_hi;
        if (!coupled && q < 2) {
          const int mpr = L.crow.d;
          t_lo = (lo - 1) * mpr;
          t_hi = (hi - 1) * mpr;
        } else {
          const ColourSlots cs = vanka_slots(L, coupled ? q : q - 2);
          const int r1 = hi - 1;  // rows lo .. r1
          if (r1 < cs.j0) continue;
          const int qlo = lo > cs.j0 ? (lo - cs.j0 + cs.rstep - 1) / cs.rstep : 0;
          const int qhi = (r1 - cs.j0) / cs.rstep;
          t_lo = qlo * cs.mpr;
          t_hi = std::min((qhi + 1) * cs.mpr, cs.n);
        }
        if (t_lo >= t_hi) continue;
        S.q[S.n] = q;
        S.t_lo[S.n] = t_lo;
        S.t_hi[S.n] = t_hi;
        S.boff[S.n] = nb;
        nb += (t_hi - t_lo + SNT - 1) / SNT;
        ++S.n;
      }
      S.boff[S.n] = nb;
      if (S.n == 0) continue;
      if (coupled) qlaunch(&k_skew<R, Form, true>, nb, SNT, 0, s, P, L, S, omega);
      else qlaunch(&k_skew<R, Form, false>, nb, SNT, 0, s, P, L, S, omega);
      ++g_launches;
      ++launches;
    }
  }
  return launches;
}

void launch_predict(double* const x[5], double* const a[5], double* const b[5],
                    double* const c[5], const double w[3], size_t n, int off, cudaStream_t s) {
  FiveArrays X, A, B, C;
  for (int q = 0; q < 5; ++q) {
    X.p[q] = x[q];
    A.p[q] = a[q];
    B.p[q] = b[q];
    C.p[q] = c[q];
  }
  const int NT = 256;
  dim3 grid((unsigned)((n + NT - 1) / NT), 5);
  qlaunch(&k_predict, grid, NT, 0, s, X, A, B, C, w[0], w[1], w[2], (long long)n, off);
  ++g_launches;
}

void launch_loop_clock(double* ctl, cudaStream_t s) {
  qlaunch(&k_loop_clock, 1, 1, 0, s, ctl);
  ++g_launches;
}
void launch_loop_ctl(const double* nrm, double* ctl, cudaGraphConditionalHandle hl,
                     cudaGraphConditionalHandle hc, double tol, int maxcyc, int diverge,
                     double limit_ns, int first, cudaStream_t s) {
  qlaunch(&k_loop_ctl, 1, 1, 0, s, nrm, ctl, hl, hc, tol, maxcyc, diverge, limit_ns, first);
  ++g_launches;
}

int partial_rows_needed(int m1, int m2) {
  dim3 g = grid2(m1 + 1, m2 + 1);
  return g.x * g.y;
}

#define QN_INSTANTIATE_FORM(T, F)                                                                \
  template int launch_coarse_vcycle<T, F>(const Prm<T>&, const Lv<T>*, int, int, int, int,        \
                                          T, int, cudaStream_t, int, int, int);                  \
  template void launch_coupled<T, F>(const Prm<T>&, const Lv<T>&, int, T, cudaStream_t, int);     \
  template void launch_residual<T, F>(const Prm<T>&, const Lv<T>&, double*, cudaStream_t);       \
  template void launch_add_op<T, F>(const Prm<T>&, const Lv<T>&, cudaStream_t);                  \
  template void launch_ch<T, F>(const Prm<T>&, const Lv<T>&, int, cudaStream_t, int);            \
  template void launch_vanka<T, F>(const Prm<T>&, const Lv<T>&, int, T, cudaStream_t, int, int, int, int);

#define QN_INSTANTIATE(T)                                                                        \
  template void launch_cast_frozen<T>(const Lv<double>&, const Lv<T>&, cudaStream_t);            \
  template void launch_start_correction<T>(const Prm<T>&, const Lv<double>&, const Lv<T>&,       \
                                           cudaStream_t);                                        \
  template void launch_apply_correction<T>(const Prm<double>&, const Lv<double>&, const Lv<T>&,    \
                                            cudaStream_t);                                          \
  template void launch_restrict_base<T>(const Prm<T>&, const Lv<T>&, const Lv<T>&, cudaStream_t); \
  template void launch_bc_unknowns<T>(const Lv<T>&, cudaStream_t);                               \
  template void launch_frozen<T>(const Prm<T>&, const Lv<T>&, cudaStream_t);                     \
  template void launch_restrict<T>(const Prm<T>&, const Lv<T>&, const Lv<T>&, cudaStream_t);      \
  template void launch_restrict_frozen<T>(const Lv<T>&, const Lv<T>&, cudaStream_t);             \
  template void launch_prolong<T>(const Prm<T>&, const Lv<T>&, const Lv<T>&, cudaStream_t);        \
  template void launch_gauge<T>(const Lv<T>&, double*, double*, cudaStream_t);                   \
  template void launch_norms_finalize<T>(const Lv<T>&, double*, double*, cudaStream_t);          \
  template void launch_mass<T>(const Prm<T>&, const Lv<T>&, const T*, double*, double*,          \
                               cudaStream_t);                                                    \
  template void launch_energy<T>(const Prm<T>&, const Lv<T>&, const T*, const T*, const T*,      \
                                 double, double, double, double*, double*, cudaStream_t);        \
  template void launch_dissipation<T>(const Prm<T>&, const Lv<T>&, double, double, double,       \
                                      double*, double*, cudaStream_t);                           \
  template void launch_pack_in<T>(const Lv<T>&, T*, const double*, int, cudaStream_t);           \
  template void launch_pack_out<T>(const Lv<T>&, double*, const T*, int, cudaStream_t);

QN_INSTANTIATE(double)
QN_INSTANTIATE(float)
QN_INSTANTIATE_FORM(double, FullForm)
QN_INSTANTIATE_FORM(double, ErrForm)
QN_INSTANTIATE_FORM(float, ErrForm)
template void launch_wave<float, ErrForm>(const Prm<float>&, const Lv<float>&, const WavePlan&,
                                          float, unsigned*, double*, cudaStream_t);
template void launch_wave<double, ErrForm>(const Prm<double>&, const Lv<double>&, const WavePlan&,
                                           double, unsigned*, double*, cudaStream_t);
template int launch_skew<float, ErrForm>(const Prm<float>&, const Lv<float>&, int, int, int, float,
                                         cudaStream_t);
template int launch_skew<double, ErrForm>(const Prm<double>&, const Lv<double>&, int, int, int, double,
                                          cudaStream_t);
// projection method (FP64, per-level launches)
template void launch_residual<double, ProjForm>(const Prm<double>&, const Lv<double>&, double*,
                                                cudaStream_t);
template int launch_coarse_vcycle<double, ProjForm>(const Prm<double>&, const Lv<double>*, int, int,
                                                    int, int, double, int, cudaStream_t, int,
                                                    int, int);
template void launch_add_op<double, ProjForm>(const Prm<double>&, const Lv<double>&, cudaStream_t);
template void launch_ch<double, ProjForm>(const Prm<double>&, const Lv<double>&, int, cudaStream_t,
                                          int);
template void launch_vanka4<double, ProjForm>(const Prm<double>&, const Lv<double>&, int, double,
                                               cudaStream_t, int);
template void launch_pgs<double>(const Prm<double>&, const Lv<double>&, int, cudaStream_t, int);
template void launch_proj_velocity<double>(const Prm<double>&, const Lv<double>&, double*, double*,
                                           cudaStream_t);
template void launch_proj_diss<double>(const Prm<double>&, const Lv<double>&, const double*,
                                       const double*, double*, double*, cudaStream_t);

}  // namespace qn
