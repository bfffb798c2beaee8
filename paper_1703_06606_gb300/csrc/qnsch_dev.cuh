// qnsch_dev.cuh -- device data structures and the discrete operator of the
// primitive method (Guo, Lin, Lowengrub & Wise, arXiv:1703.06606, Sec. 6.1) on
// the staggered grid of Sec. 5 / App. A, for sm_103a.
//
// Layout: every array of a level lives in one padded 2-D index space with one
// ghost layer: entry (I, J), I = -1..m1+1, J = -1..m2+1, at origin[J*pitch + I];
// pitch is a multiple of 32 elements so that rows start 256-byte aligned.
//   cell (i,j)        -> (i, j)       i, j = 0..m1+1 / 0..m2+1 (with ghosts)
//   u_{i+1/2, j}      -> (i, j)       i = -1..m1+1
//   v_{i, j+1/2}      -> (i, j)       j = -1..m2+1
// A thread working at cell (i,j) therefore reads cell, u and v arrays at the same
// offset plus small constant displacements.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <type_traits>

namespace qn {

// FP32 and FP64 numbers whose multiply-adds are fused by the way an expression
// is written.  The compiler contracts a * b + c as it sees fit in each kernel
// it inlines a function into; two kernels that run the same visits (a colour
// launch, the wavefront, the skewed chunks, the fused coarse V-cycle) then
// differ by rounding.  Here a product is held as its two factors until it is
// added (fused) or used (rounded): product + product fuses the left one.
template <typename F>
struct Fused {
  F v;
  Fused() = default;
  __host__ __device__ constexpr Fused(float x) : v((F)x) {}
  __host__ __device__ constexpr Fused(double x) : v((F)x) {}
  __host__ __device__ constexpr Fused(int x) : v((F)x) {}
  __host__ __device__ explicit operator float() const { return (float)v; }
  __host__ __device__ explicit operator double() const { return (double)v; }
};
typedef Fused<float> rf32;
typedef Fused<double> rf64;
static_assert(sizeof(rf32) == 4 && sizeof(rf64) == 8 && std::is_trivially_copyable<rf32>::value &&
                  std::is_trivially_copyable<rf64>::value,
              "the bits of a float and a double");
// the same bits as an object of the kernel's type: a copy, since an object may
// not be read as one of another class
template <typename R, template <typename> class S, typename T>
inline S<R> as_compute(const S<T>& x) {
  static_assert(sizeof(S<T>) == sizeof(S<R>) && std::is_trivially_copyable<S<T>>::value &&
                    std::is_trivially_copyable<S<R>>::value,
                "one layout");
  S<R> y;
  std::memcpy(static_cast<void*>(&y), &x, sizeof(y));
  return y;
}
#ifdef __CUDACC__
#define QN_F __device__ __forceinline__
QN_F float rn_add(float x, float y) { return __fadd_rn(x, y); }
QN_F float rn_mul(float x, float y) { return __fmul_rn(x, y); }
QN_F float rn_fma(float x, float y, float z) { return __fmaf_rn(x, y, z); }
QN_F double rn_add(double x, double y) { return __dadd_rn(x, y); }
QN_F double rn_mul(double x, double y) { return __dmul_rn(x, y); }
QN_F double rn_fma(double x, double y, double z) { return __fma_rn(x, y, z); }
template <typename F>
struct Product {
  F a, b;
  QN_F operator Fused<F>() const { return rn_mul(a, b); }
};
#define QN_T template <typename F> QN_F
QN_T Fused<F> operator+(Fused<F> x, Fused<F> y) { return rn_add(x.v, y.v); }
QN_T Fused<F> operator-(Fused<F> x, Fused<F> y) { return rn_add(x.v, -y.v); }
QN_T Fused<F> operator-(Fused<F> x) { return -x.v; }
QN_T Product<F> operator*(Fused<F> x, Fused<F> y) { return {x.v, y.v}; }
QN_T Product<F> operator*(Product<F> x, Fused<F> y) { return {rn_mul(x.a, x.b), y.v}; }
QN_T Product<F> operator*(Fused<F> x, Product<F> y) { return {x.v, rn_mul(y.a, y.b)}; }
QN_T Product<F> operator*(Product<F> x, Product<F> y) {
  return {rn_mul(x.a, x.b), rn_mul(y.a, y.b)};
}
QN_T Product<F> operator-(Product<F> x) { return {-x.a, x.b}; }
QN_T Fused<F> operator+(Product<F> x, Fused<F> y) { return rn_fma(x.a, x.b, y.v); }
QN_T Fused<F> operator+(Fused<F> x, Product<F> y) { return rn_fma(y.a, y.b, x.v); }
QN_T Fused<F> operator-(Product<F> x, Fused<F> y) { return rn_fma(x.a, x.b, -y.v); }
QN_T Fused<F> operator-(Fused<F> x, Product<F> y) { return rn_fma(-y.a, y.b, x.v); }
QN_T Fused<F> operator+(Product<F> x, Product<F> y) { return rn_fma(x.a, x.b, rn_mul(y.a, y.b)); }
QN_T Fused<F> operator-(Product<F> x, Product<F> y) { return rn_fma(x.a, x.b, -rn_mul(y.a, y.b)); }
QN_T Fused<F>& operator+=(Fused<F>& x, Fused<F> y) { return x = x + y; }
QN_T Fused<F>& operator-=(Fused<F>& x, Fused<F> y) { return x = x - y; }
QN_T Fused<F>& operator+=(Fused<F>& x, Product<F> y) { return x = x + y; }
QN_T Fused<F>& operator-=(Fused<F>& x, Product<F> y) { return x = x - y; }
QN_T Fused<F>& operator*=(Fused<F>& x, Fused<F> y) { return x = x * y; }
QN_T Fused<F> operator/(Fused<F> x, Fused<F> y) { return x.v / y.v; }
#undef QN_T
// the value of the lane whose index differs from this one's by the bits o
template <typename T>
QN_F T shfl_xor(T x, int o) {
  return __shfl_xor_sync(0xffffffffu, x, o);
}
template <typename F>
QN_F Fused<F> shfl_xor(Fused<F> x, int o) {
  return __shfl_xor_sync(0xffffffffu, x.v, o);
}
// lane src's value
template <typename F>
QN_F Fused<F> shfl_from(Fused<F> x, int src) {
  return __shfl_sync(0xffffffffu, x.v, src);
}
#undef QN_F
#endif

template <typename T>
struct Prm {
  T ia, ib;        // rho(c) = 1 / (ia c + ib): ia = alpha = (rho2-rho1)/(rho1 rho2), ib = 1/rho2
  T va, vb;        // viscosity mu(c) = 1 / (va c + vb)
  T alpha;         // (rho2 - rho1) / (rho1 rho2), Sec. 2.1
  T K, Lam;        // M eta/(eps We) and eps eta M/We, coefficients of (pm-num-chem)
  T iM, iRe, iPe;  // 1/M, 1/Re, 1/Pe
  T Fr_inv;        // 1/Fr (0: no gravity)
  T eps_m;         // mobility regularisation, m(c) = sqrt(c^2 (1-c)^2 + eps_m)
  T idt;           // 1/dt
};

// n / d for 0 <= n < 2^31 by one multiply-high and a shift: with s = ceil(log2
// d) - 1 and m = ceil(2^(32+s) / d), m d exceeds 2^(32+s) by less than d <=
// 2^(s+1), so the quotient's error n (m d - 2^(32+s)) / (d 2^(32+s)) stays
// below 1/d.  A run-time division takes about 25 dependent instructions, and a
// visit's slot-to-cell mapping needs three.
struct FastDiv {
  unsigned m;
  int s, d;
#ifdef __CUDACC__
  __device__ __forceinline__ int div(int n) const {
    return d == 1 ? n : (int)(__umulhi((unsigned)n, m) >> s);
  }
#endif
};
inline FastDiv fast_div(int d) {
  int s = -1;
  while ((1LL << (s + 1)) < d) ++s;
  if (s < 0) return {0u, 0, 1};
  return {(unsigned)(((1ULL << (32 + s)) + (unsigned)d - 1) / (unsigned)d), s, d};
}

// Products of the parameters and a level's spacing that the operators multiply
// by (level_consts, on the host at each launch).  A warp's FP64 instruction
// holds its sub-partition's pipe for 64 to 76 cycles whether its operands vary
// by lane or not, so a product of two kernel parameters costs a visit as much
// as one of its own terms; formed here it costs nothing.
template <typename T>
struct LvK {
  T qidt;              // 1/(4 dt): A rho(c) / (2 dt) from the sum of the edge's two densities
  T ihM;               // 1/(M h)
  T v1, v3;            // 1/(Re h^2), a third of it
  T hih;               // 1/(2 h)
  T dif, adif, a2dif;  // 1/(2 Pe h^2), alpha and alpha^2 times it
  T ihaM;              // 1/(M h^2)
  T hih2;              // 1/(2 h^2)
  T K8, K4;            // K/8, K/4
  T L4, L8, L4h;       // Lam/4, Lam/(8 h^2), Lam/(4 h^2)
  T kick, hkick, gdt;  // 2 dt/(M h), half of it, dt/Fr: the projection equation
  T pdiv;              // 2 dt/(M h^2): its derivative in the pressure
};

template <typename T>
struct Lv {
  typedef T real;
  static constexpr bool has_rho = true;  // rhoc may be set
  static constexpr bool all_arrays = true;  // also those that only some kernels read
  LvK<T> k;
  // slot-to-cell mapping: cells of a Vanka colour in one of its rows, of a CH
  // colour in a row, and the number of Vanka colours
  FastDiv vrow, crow, kdiv;
  long long nst;  // elements from one array of the level to the next
  int m1, m2, px, pitch;
  // Vanka colours of this level: kcol colours, (2i+j) mod 8 when c8 is set
  // (periodic x with m1 = 0 mod 4), else (i+2j) mod kcol
  int kcol, c8;
  T h, ih, ih2;
  T *c, *mu, *p, *u, *v;       // iterate
  T *fc, *fmu, *fp, *fu, *fv;  // FAS right-hand side
  T *rc, *rmu, *rp, *ru, *rv;  // residual f - N(x)
  T *sc, *smu, *sp, *su, *sv;  // restricted iterate kept for the correction
  T *cn, *un, *vn;             // frozen level-n data
  T *rhon, *mobn, *visn, *Gn;  // rho(c^n), m(c^n), mu(c^n), G(c^n)
  // coefficients of (pm-num-mx) that depend on frozen data only, built once
  // per step: A_x rho^n, A_y rho^n (edges); rho^n a_x u^n, rho^n a_y v^n
  // (cells); Acal rho^n Acal_x v^n, Acal rho^n Acal_y u^n, Acal mu(c^n)
  // (vertices (i+1/2, j+1/2) at (i,j)); D_x c^n / 2, D_y c^n / 2 (edges);
  // the divergence corrections 1/2[D_x(rho a_x u) + Dfrak_y(..)] (x-edges)
  // and 1/2[Dfrak_x(..) + D_y(rho a_y v)] (y-edges) of (e1e1-2)
  T *Aru, *Arv, *Sx, *Sy, *Qx, *Qy, *Av, *Tx, *Ty, *Dvu, *Dvv;
  // built per step (they depend on dt): for each
  // momentum row (x-edges *u, y-edges *v) the time-term coefficients, time =
  // x T1 + T0 + (dt^-1/2) A rho(c) x with T1 = A rho^n/(2dt) + Dv and T0 =
  // -A rho^n x^n/dt (plus, in the primitive method's y rows, gravity
  // (1/Fr) A_y rho^n), and, on the full-iterate levels, Dg, the part of the row's diagonal entry that does not
  // depend on the iterate (the whole diagonal is Dg + A rho(c)/(2dt))
  T *T1u = nullptr, *T1v = nullptr, *T0u = nullptr, *T0v = nullptr, *Dgu = nullptr, *Dgv = nullptr;
  // FP64 full-iterate levels only: rho(c) of the iterate, ghosts included.
  // Every kernel that writes c writes rho(c) beside it, so the smoothers and
  // the residual read the density instead of dividing for it; the values are
  // those rho_of gives.
  T* rhoc = nullptr;
  // FP64 full-iterate levels only, built per step: the momentum rows of
  // (pm-num-mx) assembled as stencils.  Apart from the density term A rho(c)
  // u / (2dt), each row is linear in the iterate with coefficients that depend
  // on frozen data only.  For the x row at edge k (y row: u <-> v, strides
  // swapped): Cu multiplies u at the edge itself, aPu / aMu its neighbours
  // along x (k + 1, k - 1), tPu / tMu across (k + W, k - W), M0u / M1u the mu of
  // the cells k and k + 1.  Wall edges read their reflected ghosts, as the
  // unassembled row does.
  T *Cu = nullptr, *aPu = nullptr, *aMu = nullptr, *tPu = nullptr, *tMu = nullptr,
    *M0u = nullptr, *M1u = nullptr;
  T *Cv = nullptr, *aPv = nullptr, *aMv = nullptr, *tPv = nullptr, *tMv = nullptr,
    *M0v = nullptr, *M1v = nullptr;
  // error-equation (defect-correction) levels only: base state X the iterate
  // e is a correction to, and X.c - c^n formed in FP64 before rounding
  T *Bc = nullptr, *Bmu = nullptr, *Bu = nullptr, *Bv = nullptr, *Bdc = nullptr;
  T* rB = nullptr;  // rho(Bc)
  __device__ __forceinline__ int at(int i, int j) const { return j * pitch + i; }
  // the array of direction d (0: x, 1: y) of a pair
  // (the pairs' arrays are neighbours, the assembled rows' seven apart): an
  // offset, where selecting between two kernel parameters is an indexed
  // constant load that the array's own load has to wait for
  __device__ __forceinline__ T* pair(int d, T* x, T*) const { return x + (d ? nst : 0); }
  __device__ __forceinline__ T* row_pair(int d, T* x, T*) const { return x + (d ? 7 * nst : 0); }
  // x-edge unknowns: walls exclude i = 0 and i = m1; periodic keeps i = m1 (= edge 0)
  __device__ __forceinline__ int uhi() const { return px ? m1 : m1 - 1; }
};

// a b / d rounded once: the remainders of the product and of the quotient are
// exact.  A constant's rounding is in every cell, so that a product of three
// that rounds at each would cost what folding it saves in a cell's own.
inline double mul_div(double a, double b, double d) {
  const double p = a * b, q = p / d;
  return std::isfinite(q) ? q + (std::fma(-q, d, p) + std::fma(a, b, -p)) / d : q;
}

// L with its constants for the parameters P
template <typename T>
inline Lv<T> level_consts(const Prm<T>& P, const Lv<T>& L) {
  const double ih = L.ih, ih2 = L.ih2, iM = P.iM, dif = 0.5 * P.iPe * ih2, al = P.alpha;
  const double hkick = mul_div(ih, iM, P.idt);
  Lv<T> X = L;
  X.k = {T(0.25 * P.idt), T(ih * iM),       T(P.iRe * ih2),         T(P.iRe * ih2 / 3.0),
         T(0.5 * ih),     T(dif),           T(al * dif),            T(al * al * dif),
         T(ih * ih * iM), T(0.5 * ih2),     T(0.125 * P.K),         T(0.25 * P.K),
         T(0.25 * P.Lam), T(0.125 * P.Lam * ih2), T(0.25 * P.Lam * ih2),
         T(2.0 * hkick),  T(hkick),         T(P.Fr_inv / P.idt),
         T(2.0 * ih2 * iM / P.idt)};
  X.vrow = fast_div(L.c8 ? (L.m1 + 3) / 4 : (L.m1 + L.kcol - 1) / L.kcol);
  X.crow = fast_div((L.m1 + 1) / 2);
  X.kdiv = fast_div(L.kcol);
  return X;
}

// The arrays of an FP64 full-iterate level in the order in which they sit in
// the level's block (one allocation, NFIELD arrays of the same padded size):
// X(member) for each.
#define QN_LV_ARRAYS(X)                                                                        \
  X(c) X(mu) X(p) X(u) X(v) X(fc) X(fmu) X(fp) X(fu) X(fv) X(rc) X(rmu) X(rp) X(ru) X(rv)     \
  X(sc) X(smu) X(sp) X(su) X(sv) X(cn) X(un) X(vn) X(rhon) X(mobn) X(visn) X(Gn) X(Aru)       \
  X(Arv) X(Sx) X(Sy) X(Qx) X(Qy) X(Av) X(Tx) X(Ty) X(Dvu) X(Dvv) X(T1u) X(T1v) X(T0u) X(T0v)  \
  X(Dgu) X(Dgv) X(rhoc) X(Cu) X(aPu) X(aMu) X(tPu) X(tMu) X(M0u) X(M1u) X(Cv) X(aPv) X(aMv)   \
  X(tPv) X(tMv) X(M0v) X(M1v)

// ---------------------------------------------------------------------------
// constitutive functions (Sec. 2.1) and secants (Sec. 4.1)
// ---------------------------------------------------------------------------
template <typename T> __device__ __forceinline__ T rho_of(const Prm<T>& P, T c) {
  return T(1) / (P.ia * c + P.ib);
}
// a / b: in FP32 (the error-equation smoothers) the fast division, within 2
// ulp, whose rounding the FP64 defect correction absorbs; IEEE division in FP64
template <typename T> __device__ __forceinline__ T qdiv(T a, T b) { return a / b; }
template <> __device__ __forceinline__ float qdiv(float a, float b) { return __fdividef(a, b); }
template <> __device__ __forceinline__ rf32 qdiv(rf32 a, rf32 b) { return __fdividef(a.v, b.v); }
// 1/x for the pivots of the local block solves.  FP32: the fast division, as
// qdiv.  FP64: one step of the third-order iteration r <- r + r (e + e^2),
// e = 1 - x r, which is Newton's for the zero of 1/r - x with the next term of
// the geometric series 1/(1 - e) kept, so the relative error e of r becomes
// e^3; started from the hardware's approximate reciprocal
// (rcp.approx.ftz.f64) the result is within a few units in the last place of
// 1/x (tested against IEEE division) in three FP64 instructions, where two
// Newton steps take four and the division 1/x five.  Normal-range x only:
// the pivots are determinants and diagonal sums of the local systems, far from
// the subnormal range.  Not for a density: its error reaches 0.5065 units (6e6
// arguments; 3 in 10^4 differ from the division), and rho(c) is a term of the
// rows themselves, so rho_of divides, in FP64 with the division's rounding.
template <typename T> __device__ __forceinline__ T qrcp(T x) { return qdiv(T(1), x); }
template <> __device__ __forceinline__ double qrcp(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  double e = __fma_rn(-x, r, 1.0);
  e = __fma_rn(e, e, e);
  return __fma_rn(r, e, r);
}
template <> __device__ __forceinline__ rf64 qrcp(rf64 x) { return qrcp(x.v); }
template <> __device__ __forceinline__ float rho_of(const Prm<float>& P, float c) {
  return qdiv(1.0f, P.ia * c + P.ib);
}
template <> __device__ __forceinline__ rf32 rho_of(const Prm<rf32>& P, rf32 c) {
  return qdiv(rf32(1.0f), P.ia * c + P.ib);
}
template <typename T> __device__ __forceinline__ T visc_of(const Prm<T>& P, T c) {
  return T(1) / (P.va * c + P.vb);
}
template <typename T> __device__ __forceinline__ T mob_of(const Prm<T>& P, T c) {
  T w = c * (T(1) - c);
  return sqrt(w * w + P.eps_m);
}
template <typename T> __device__ __forceinline__ T Fdw(T c) {
  T w = c * (c - T(1));
  return T(0.25) * w * w;
}
template <typename T> __device__ __forceinline__ T fdw(T c) { return c * (c - T(1)) * (c - T(0.5)); }
// g(a,b) with F(a) - F(b) = g(a,b) (a - b)
template <typename T> __device__ __forceinline__ T gsec(T a, T b) {
  return T(0.25) * (a * (a - T(1)) + b * (b - T(1))) * (a + b - T(1));
}
template <typename T> __device__ __forceinline__ T gsec_da(T a, T b) {
  return T(0.25) * ((T(2) * a - T(1)) * (a + b - T(1)) + a * (a - T(1)) + b * (b - T(1)));
}

// ---------------------------------------------------------------------------
// pieces of the discrete operator N(x) (Sec. 6.1)
// ---------------------------------------------------------------------------

// G(c) = a_x((D_x c)^2) + a_y((D_y c)^2) at cell k (times h^2)
template <class A>
__device__ __forceinline__ auto G_h2(A c, int k, int pitch) ->
    typename std::decay<decltype(c[k])>::type {
  typedef typename std::decay<decltype(c[k])>::type T;
  T cc = c[k];
  T de = c[k + 1] - cc, dw = cc - c[k - 1], dn = c[k + pitch] - cc, ds = cc - c[k - pitch];
  return T(0.5) * (de * de + dw * dw + dn * dn + ds * ds);
}

// Momentum row d (0: x row at x-edge k, unknown u; 1: y row at y-edge k,
// unknown v) of (pm-num-mx), with (e1e1-1), (e1e1-2) and (e1e1), from the
// per-step assembled stencil (the arrays Cu.. / Cv.. of Lv): the row's terms
// regrouped by unknown.  rs = the sum of rho(c) over the edge's two cells.  s
// is the stride along the edge normal, t across it; a the row's own velocity, b
// the other one.
template <typename T, class LV>
__device__ __forceinline__ T mom_asm(const LV& L, int d, int k, T rs) {
  const int s = d ? L.pitch : 1, t = d ? 1 : L.pitch;
  auto a = L.pair(d, L.u, L.v);
  auto b = L.pair(1 - d, L.u, L.v);
  auto C = L.row_pair(d, L.Cu, L.Cv);
  auto aP = L.row_pair(d, L.aPu, L.aPv);
  auto aM = L.row_pair(d, L.aMu, L.aMv);
  auto tP = L.row_pair(d, L.tPu, L.tPv);
  auto tM = L.row_pair(d, L.tMu, L.tMv);
  T r = L.pair(d, L.T0u, L.T0v)[k] + (C[k] + L.k.qidt * rs) * a[k];
  r += aP[k] * a[k + s] + aM[k] * a[k - s] + tP[k] * a[k + t] + tM[k] * a[k - t];
  // the grad-div term's cross derivative of the other velocity
  T vl = L.visn[k], vr = L.visn[k + s];
  r -= L.k.v3 * (vr * (b[k + s] - b[k + s - t]) - vl * (b[k] - b[k - t]));
  r += (L.p[k + s] - L.p[k]) * L.k.ihM + L.row_pair(d, L.M0u, L.M0v)[k] * L.mu[k] +
       L.row_pair(d, L.M1u, L.M1v)[k] * L.mu[k + s];
  return r;
}

// The intermediate velocity's row (pj-num-mx) of the projection method: no
// pressure and no surface tension, and T0 without gravity (that acts in the
// projection equation).  From the fluxes' unscaled differences: 25 FP64
// instructions where the assembled stencil would take 11, but the stencil's
// products round at a / h^2 and the differences at (a's difference) / h^2
// (256 cells across, viscosity ratio 20, dt 3e-4: 5.8e-14 against 1.0e-11 of a
// row of size 1e4; the scaled differences of the equation as written 7.0e-14).
template <typename T, class LV>
__device__ __forceinline__ T proj_mom_row(const LV& L, int d, int k, T rs) {
  const int s = d ? L.pitch : 1, t = d ? 1 : L.pitch;
  auto a = L.pair(d, L.u, L.v);
  auto b = L.pair(1 - d, L.u, L.v);
  auto S = L.pair(d, L.Sx, L.Sy);
  auto Q = L.pair(d, L.Qx, L.Qy);
  T ae = a[k], vl = L.visn[k], vr = L.visn[k + s];
  T dl = ae - a[k - s], dr = a[k + s] - ae, dm = ae - a[k - t], dp = a[k + t] - ae;
  T el = dl + (b[k] - b[k - t]), er = dr + (b[k + s] - b[k + s - t]);
  T r = L.pair(d, L.T0u, L.T0v)[k] + L.pair(d, L.T1u, L.T1v)[k] * ae;
  r += L.k.qidt * rs * ae;
  r += L.k.hih * (S[k + s] * dr + S[k] * dl + Q[k] * dp + Q[k - t] * dm);
  r -= L.k.v1 * ((vr * dr - vl * dl) + (L.Av[k] * dp - L.Av[k - t] * dm));
  r -= L.k.v3 * (vr * er - vl * el);
  return r;
}
// the full iterate's momentum row of either method
template <bool PROJ, typename T, class LV>
__device__ __forceinline__ T full_mom_row(const LV& L, int d, int k, T rs) {
  if constexpr (PROJ) return proj_mom_row(L, d, k, rs);
  else return mom_asm(L, d, k, rs);
}

// ---------------------------------------------------------------------------
// projection method (Sec. 6.2): the iterate's u, v arrays hold the
// intermediate velocity; the new velocity follows from the projection
// equation (pj-num-pjx), A rho(c) (u - ut)/dt = -(1/M) D p + (1/M) ST(c, mu)
// [- (1/Fr) A_y rho(c) in y], ST the surface-tension pairing of (e1e1) at
// level n+1.  Gravity acts here, tested with u^{n+1} in the energy proof.
// ---------------------------------------------------------------------------
// what the projection adds to the velocity of the face between cells a and b,
// without gravity: (ST - D p) dt / (M A rho), from both cells' rho and mu, the
// differences of c and p, with the constants folded and one reciprocal (rms
// error 0.98e-16 of its terms; scaled step by step and divided 1.05e-16)
template <typename T, class LV>
__device__ __forceinline__ T proj_kick(const LV& L, T ra, T rb, T mua, T mub, T dc, T dp) {
  return (L.k.hkick * ((rb * mua + ra * mub) * dc) - L.k.kick * dp) * qrcp(ra + rb);
}
// u^{n+1} at edge (i+1/2, j), i = 0..m1; zero on no-slip walls
template <typename T, class LV>
__device__ __forceinline__ T proj_u(const Prm<T>& P, const LV& L, int i, int j) {
  if (!L.px && (i <= 0 || i >= L.m1)) return T(0);
  int k = L.at(i, j);
  T cl = L.c[k], cr = L.c[k + 1];
  return L.u[k] + proj_kick(L, rho_of(P, cl), rho_of(P, cr), L.mu[k], L.mu[k + 1], cr - cl,
                            L.p[k + 1] - L.p[k]);
}
// v^{n+1} at edge (i, j+1/2), j = 0..m2; zero on the walls in y
template <typename T, class LV>
__device__ __forceinline__ T proj_v(const Prm<T>& P, const LV& L, int i, int j) {
  if (j <= 0 || j >= L.m2) return T(0);
  const int W = L.pitch;
  int k = L.at(i, j);
  T cb = L.c[k], ct = L.c[k + W];
  return L.v[k] + proj_kick(L, rho_of(P, cb), rho_of(P, ct), L.mu[k], L.mu[k + W], ct - cb,
                            L.p[k + W] - L.p[k]) - L.k.gdt;
}
// The four face velocities u^{n+1} of cell (i,j) (E, W, N, S), from rho(c) of the
// cell (rk) and of its neighbours (rq[f] for k + 1, k - 1, k + W, k - W): the
// same values as proj_u / proj_v without re-evaluating the densities.
template <typename T, class LV>
__device__ __forceinline__ void proj_faces(const Prm<T>& P, const LV& L, int i, int j, T rk,
                                           const T (&rq)[4], T (&w)[4]) {
  const int W = L.pitch;
  int k = L.at(i, j);
  auto c = L.c;
  auto mu = L.mu;
  auto p = L.p;
  // face between cells a (left/below) and b = a + off, velocity array at a
  auto face = [&](int a, int off, auto vel, T ra, T rb) {
    return vel[a] + proj_kick(L, ra, rb, mu[a], mu[a + off], c[a + off] - c[a], p[a + off] - p[a]);
  };
  w[0] = (!L.px && i == L.m1) ? T(0) : face(k, 1, L.u, rk, rq[0]);
  w[1] = (!L.px && i == 1) ? T(0) : face(k - 1, 1, L.u, rq[1], rk);
  w[2] = (j == L.m2) ? T(0) : face(k, W, L.v, rk, rq[2]) - L.k.gdt;
  w[3] = (j == 1) ? T(0) : face(k - W, W, L.v, rq[3], rk) - L.k.gdt;
}
// (pj-num-phase): rho^n (c - c^n)/dt + a_x(rho_ew D_x c u^{n+1}) + a_y(...)
// - (1/Pe) grad_d.(A m^n grad_D mu) - (alpha/Pe) grad_d.(A m^n grad_D p), with
// rho = rho(c^{n+1}) and c^{n+1} in the advection; and (pj-num-mass): d_x u^{n+1}
// + d_y v^{n+1} - (alpha/Pe)(grad.(A m grad mu) + alpha grad.(A m grad p)).
// Both from the shared densities rq and the face velocities w of proj_faces.
// flux: the face sum of (m(c^n) of both cells) (d mu + alpha d p)
template <typename T, class LV>
__device__ __forceinline__ T opp_c_w(const Prm<T>& P, const LV& L, int k, const T (&rq)[4],
                                     const T (&w)[4], T flux) {
  const int W = L.pitch;
  auto c = L.c;
  T ck = c[k];
  T adv = rq[0] * (c[k + 1] - ck) * w[0] + rq[1] * (ck - c[k - 1]) * w[1] +
          rq[2] * (c[k + W] - ck) * w[2] + rq[3] * (ck - c[k - W]) * w[3];
  return L.rhon[k] * (ck - L.cn[k]) * P.idt + L.k.hih * adv - L.k.dif * flux;
}
template <typename T, class LV>
__device__ __forceinline__ T opp_p_w(const LV& L, const T (&w)[4], T flux) {
  return (w[0] - w[1] + w[2] - w[3]) * L.ih - L.k.adif * flux;
}

// ---------------------------------------------------------------------------
// stores that keep ghost copies consistent (App. A.6 boundary conditions)
// ---------------------------------------------------------------------------
template <typename T, class LV, class A>
__device__ __forceinline__ void store_cell(const LV& L, A a, int i, int j, T x) {
  const int W = L.pitch;
  int k = j * W + i;
  a[k] = x;
  if (i == 1) a[k + (L.px ? L.m1 : -1)] = x;       // ghost (m1+1, j) or (0, j)
  if (i == L.m1) a[k + (L.px ? -L.m1 : 1)] = x;    // ghost (0, j) or (m1+1, j)
  if (j == 1) a[k - W] = x;
  if (j == L.m2) a[k + W] = x;
}

template <typename T, class LV>
__device__ __forceinline__ void store_u(const LV& L, int e, int j, T x) {
  const int W = L.pitch;
  auto u = L.u;
  int cols[3] = {e, e, e};
  int n = 1;
  if (L.px) {
    if (e == L.m1) cols[n++] = 0;
    if (e == L.m1 - 1) cols[n++] = -1;
    if (e == 1) cols[n++] = L.m1 + 1;
  }
  for (int q = 0; q < n; ++q) {
    int k = j * W + cols[q];
    u[k] = x;
    if (j == 1) u[k - W] = -x;
    if (j == L.m2) u[k + W] = -x;
  }
}

template <typename T, class LV>
__device__ __forceinline__ void store_v(const LV& L, int i, int e, T x) {
  const int W = L.pitch;
  auto v = L.v;
  int k = e * W + i;
  v[k] = x;
  if (L.px) {
    if (i == L.m1) v[k - L.m1] = x;
    if (i == 1) v[k + L.m1] = x;
  } else {
    if (i == 1) v[k - 1] = -x;
    if (i == L.m1) v[k + 1] = -x;
  }
}

// Whether any value that a block on cell (i,j) writes has a ghost copy: only
// then do its stores go through store_cell, store_u and store_v.
template <class LV>
__device__ __forceinline__ bool has_ghosts(const LV& L, int i, int j) {
  return i <= 2 || i >= L.m1 - 1 || j == 1 || j == L.m2;
}
template <typename T, class LV, class A>
__device__ __forceinline__ void put_cell(const LV& L, A a, int i, int j, bool ghosts, T x) {
  if (ghosts) store_cell(L, a, i, j, x);
  else a[L.at(i, j)] = x;
}
// the four edges (W, E, S, N) of cell (i,j); act: the ones that hold an unknown
template <typename T, class LV>
__device__ __forceinline__ void put_edges(const LV& L, int i, int j, bool ghosts,
                                          const bool* act, T w, T e, T so, T n) {
  if (ghosts) {
    if (act[0]) store_u(L, (L.px && i == 1) ? L.m1 : i - 1, j, w);
    if (act[1]) store_u(L, i, j, e);
    if (act[2]) store_v(L, i, j - 1, so);
    if (act[3]) store_v(L, i, j, n);
  } else {
    const int k = L.at(i, j);
    L.u[k - 1] = w;
    L.u[k] = e;
    L.v[k - L.pitch] = so;
    L.v[k] = n;
  }
}
// edge q (W, E, S, N) of cell (i,j), which holds an unknown, by one lane of a team
template <typename T, class LV>
__device__ __forceinline__ void put_edge(const LV& L, int i, int j, int q, bool ghosts, T x) {
  if (ghosts) {
    if (q < 2) store_u(L, q ? i : (L.px && i == 1) ? L.m1 : i - 1, j, x);
    else store_v(L, i, q == 3 ? j : j - 1, x);
  } else {
    const int k = L.at(i, j);
    L.pair(q >> 1, L.u, L.v)[q == 0 ? k - 1 : q == 2 ? k - L.pitch : k] = x;
  }
}

// ---------------------------------------------------------------------------
// error equation for defect correction: N_e(e) = N(X + e) - N(X) for the
// iterate e stored in c, mu, p, u, v of the level and the base X in Bc, Bmu, Bu,
// Bv.  Every nonlinear difference is written with the secant identities of
// Sec. 4.1 (rho(a) - rho(b) = r(a,b)(a-b), F(a) - F(b) = g(a,b)(a-b)) and the
// algebraic factorisations below, so that no term is a difference of two
// nearly equal numbers: in FP32 the result keeps the relative accuracy of e.
// ---------------------------------------------------------------------------

// r(a,b) = -alpha rho(a) rho(b)
template <typename T> __device__ __forceinline__ T rsec_(const Prm<T>& P, T ra, T rb) {
  return -P.alpha * ra * rb;
}
// g(a+e, b) - g(a, b) = e/4 [a(a-1) + b(b-1) + (2a - 1 + e)(a + b - 1 + e)]
template <typename T> __device__ __forceinline__ T dgsec(T a, T b, T e) {
  return T(0.25) * e * (a * (a - T(1)) + b * (b - T(1)) + (T(2) * a - T(1) + e) * (a + b - T(1) + e));
}

// What the rows of the error equation at a cell share, at the cell and its east,
// west, north and south neighbours: e and the base's c and rho^n, rho at the
// full value and the difference rho(C + e) - rho(C).
template <typename T>
struct ErrCell {
  T e[5], B[5], rn[5], r[5], dr[5];
};
template <typename T, class LV>
__device__ __forceinline__ ErrCell<T> err_cell(const Prm<T>& P, const LV& L, int k) {
  const int off[5] = {0, 1, -1, L.pitch, -L.pitch};
  ErrCell<T> X;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    X.e[q] = L.c[k + off[q]];
    X.B[q] = L.Bc[k + off[q]];
    X.rn[q] = L.rhon[k + off[q]];
    X.dr[q] = L.rB[k + off[q]];
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    X.r[q] = rho_of(P, X.B[q] + X.e[q]);
    X.dr[q] = rsec_(P, X.r[q], X.dr[q]) * X.e[q];
  }
  return X;
}

// N_c of the error equation without its diffusion: (pm-num-phase) applied to e
template <typename T, class LV>
__device__ __forceinline__ T err_c(const Prm<T>& P, const LV& L, int k, T rp) {
  auto rn = L.rhon;
  const int W = L.pitch;
  T adv = rn[k + 1] * L.Tx[k] * L.u[k] + rn[k - 1] * L.Tx[k - 1] * L.u[k - 1] +
          rn[k + W] * L.Ty[k] * L.v[k] + rn[k - W] * L.Ty[k - W] * L.v[k - W];
  return L.c[k] * (rp + rsec_(P, rp, L.rB[k]) * L.Bdc[k]) * P.idt + adv;
}

// N_mu of the error equation
template <typename T, class LV>
__device__ __forceinline__ T err_mu(const Prm<T>& P, const LV& L, int k, const ErrCell<T>& X) {
  const int off[5] = {0, 1, -1, L.pitch, -L.pitch};
  T ek = X.e[0], Ck = X.B[0], cnk = L.cn[k], rnk = X.rn[0], rp = X.r[0];
  T cp = Ck + ek;
  T dr = X.dr[0];                           // rho(c') - rho(C)
  T rhp = T(0.5) * (rp + rnk);              // rho^{n+1/2} at c'
  T r_new = rsec_(P, rp, rnk);              // r(c', c^n)
  T d_r = -P.alpha * rnk * dr;              // r(c', c^n) - r(C, c^n)
  T dF = gsec(cp, Ck) * ek;                 // F(c') - F(C)
  T dbulk = rhp * dgsec(Ck, cnk, ek) + T(0.5) * dr * gsec(Ck, cnk) + T(0.5) * dF * r_new +
            T(0.5) * (Fdw(Ck) + Fdw(cnk)) * d_r;
  // G(c') - G(C) and G(C), both times 2 h^2
  T dG = T(0), GC = T(0), ddiv = T(0);
  T chP = Ck + cnk;  // 2 c^{n+1/2} at C
#pragma unroll
  for (int f = 1; f < 5; ++f) {
    T dC = X.B[f] - Ck, de = X.e[f] - ek;
    dG += de * (T(2) * dC + de);
    GC += dC * dC;
    // div(A rho_h(c') grad(e/2)) + div(A d rho_h grad c^{n+1/2}(C)), per face
    ddiv += (rhp + T(0.5) * (X.r[f] + X.rn[f])) * de +
            T(0.5) * (dr + X.dr[f]) * ((X.B[f] + L.cn[k + off[f]]) - chP);
  }
  T dgrad = L.k.L4 * (L.k.hih2 * dG * r_new + (L.k.hih2 * GC + L.Gn[k]) * d_r);
  return rp * L.mu[k] + dr * L.Bmu[k] - P.K * dbulk - dgrad + L.k.L4h * ddiv;
}

// momentum row d (0: x, 1: y) at edge k of the error equation: the terms of the
// row that are linear in (u, v, p, mu) from the per-step coefficients, over
// differences to the edge's own velocity (so that a smooth e keeps its relative
// accuracy in FP32), plus 1/2 (A rho(c') - A rho^n) e/dt and 1/2 A (rho(c') -
// rho(C)) U/dt.  rs and ds: the sums of rho(c') and of rho(c') - rho(C) over
// the edge's two cells.
template <typename T, class LV>
__device__ __forceinline__ T err_row(const Prm<T>& P, const LV& L, int d, int k, T rs, T ds) {
  const int s = d ? L.pitch : 1, t = d ? 1 : L.pitch;
  auto a = L.pair(d, L.u, L.v);
  auto b = L.pair(1 - d, L.u, L.v);
  auto rn = L.rhon;
  auto mu = L.mu;
  T ae = a[k];
  T r = (L.pair(d, L.T1u, L.T1v)[k] + L.k.qidt * rs) * ae +
        L.k.qidt * ds * L.pair(d, L.Bu, L.Bv)[k];
  r += L.pair(d, L.aPu, L.aPv)[k] * (a[k + s] - ae);
  r += L.pair(d, L.aMu, L.aMv)[k] * (a[k - s] - ae);
  r += L.pair(d, L.tPu, L.tPv)[k] * (a[k + t] - ae);
  r += L.pair(d, L.tMu, L.tMv)[k] * (a[k - t] - ae);
  T vl = L.visn[k], vr = L.visn[k + s];
  r -= L.k.v3 * (vr * (b[k + s] - b[k + s - t]) - vl * (b[k] - b[k - t]));
  r += (L.p[k + s] - L.p[k]) * L.k.ihM;
  r -= (rn[k + s] * mu[k] + rn[k] * mu[k + s]) * (L.pair(d, L.Tx, L.Ty)[k] * P.iM);
  return r;
}
// the row's diagonal entry in its own velocity; gp, gm: 2 where the neighbour
// across on that side is a wall's reflected ghost, else 1
template <typename T, class LV>
__device__ __forceinline__ T err_diag(const LV& L, int d, int k, T rs, T gp, T gm) {
  return L.pair(d, L.T1u, L.T1v)[k] + L.k.qidt * rs - L.pair(d, L.aPu, L.aPv)[k] -
         L.pair(d, L.aMu, L.aMv)[k] - gp * L.pair(d, L.tPu, L.tPv)[k] -
         gm * L.pair(d, L.tMu, L.tMv)[k];
}

// The forms of the iterate: Full (x itself, Sec. 6.1), Proj (the projection
// method on the full iterate; its u, v arrays hold the intermediate velocity)
// and Err (a correction e to the base X of a defect-correction cycle).  val_c
// .. return the full values that the local Jacobians of the smoothers are
// evaluated at, rho the density there.
struct FullForm {
  template <class LV> static __device__ __forceinline__ typename LV::real val_u(const LV& L, int k) {
    return L.u[k];
  }
  template <class LV> static __device__ __forceinline__ typename LV::real val_v(const LV& L, int k) {
    return L.v[k];
  }
  template <typename T, class LV>
  static __device__ __forceinline__ T rho(const Prm<T>&, const LV& L, int k) {
    return L.rhoc[k];
  }
};
struct ProjForm : FullForm {};
struct ErrForm {
  template <class LV> static __device__ __forceinline__ typename LV::real val_c(const LV& L, int k) {
    return L.Bc[k] + L.c[k];
  }
  template <class LV> static __device__ __forceinline__ typename LV::real val_u(const LV& L, int k) {
    return L.Bu[k] + L.u[k];
  }
  template <class LV> static __device__ __forceinline__ typename LV::real val_v(const LV& L, int k) {
    return L.Bv[k] + L.v[k];
  }
  template <class LV> static __device__ __forceinline__ typename LV::real val_mu(const LV& L, int k) {
    return L.Bmu[k] + L.mu[k];
  }
  template <typename T, class LV>
  static __device__ __forceinline__ T rho(const Prm<T>& P, const LV& L, int k) {
    return rho_of(P, val_c(L, k));
  }
};

}  // namespace qn
