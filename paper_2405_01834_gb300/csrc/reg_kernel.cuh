// Register-resident quartet kernel for small classes: one thread per shell
// quartet, every intermediate of Sec. 2 in registers (the paper's smallest
// GPU variant V0, Sec. 3, where a thread owns a whole shellset).
//
// Per thread, for every bra primitive pair and every ket primitive pair:
// Boys seeds [0]^(m) = (-2 rho)^m pref F_m(T) (Eq. 0m), the Hermite integrals
// [tuv] by Eq. r computed in place (orders high to low), and the ket
// transform [p|cd] += sum_q (-1)^|q| E^cd_q [p+q] (Eqs. pq, ket-from-hermite;
// the ket records carry the sign); after the ket primitives, the bra
// transform [ab|cd] += sum_p E^ab_p [p|cd] (Eq. bra-from-hermite). All loop
// bounds and indices are compile-time constants, so the arrays live in
// registers. Only the store and the exchange-digestion epilogues exist here;
// gradient launches use the team kernel.
#pragma once

#include <algorithm>
#include <utility>

#include "kernels.cuh"

namespace mdx {
namespace reg {

constexpr __host__ __device__ int ncart(int l) { return (l + 1) * (l + 2) / 2; }
constexpr __host__ __device__ int tet(int n) { return n < 0 ? 0 : n * (n + 1) * (n + 2) / 6; }
constexpr __host__ __device__ int tri(int n) { return n < 0 ? 0 : n * (n + 1) / 2; }
constexpr __host__ __device__ int nherm(int L) { return tet(L + 1); }
// (t,u,v) -> position in a [t][u][v] simplex of total order N (t+u+v <= N)
constexpr __host__ __device__ int hidx(int N, int t, int u, int v) {
  return tet(N + 1) - tet(N - t + 1) + tri(N - t + 1) - tri(N - t - u + 1) + v;
}
// Cartesian component k of shell l (a_x = l..0, then a_y = l-a_x..0)
constexpr __host__ __device__ int cx(int l, int k) {
  int ax = l;
  while (k > l - ax) { k -= l - ax + 1; --ax; }
  return ax;
}
constexpr __host__ __device__ int cy(int l, int k) {
  int ax = l;
  while (k > l - ax) { k -= l - ax + 1; --ax; }
  return l - ax - k;
}
constexpr __host__ __device__ int cz(int l, int k) { return l - cx(l, k) - cy(l, k); }
// per-axis E table of a record: (a,b) block start, t contiguous (library record layout)
constexpr __host__ __device__ int etab_size(int la, int lb) {
  int s = 0;
  for (int a = 0; a <= la; ++a)
    for (int b = 0; b <= lb; ++b) s += a + b + 1;
  return s;
}
constexpr __host__ __device__ int etab_off(int lb, int a, int b) {
  int s = 0;
  for (int a2 = 0; a2 < a; ++a2)
    for (int b2 = 0; b2 <= lb; ++b2) s += a2 + b2 + 1;
  for (int b2 = 0; b2 < b; ++b2) s += a + b2 + 1;
  return s;
}
constexpr __host__ __device__ int rec_size(int la, int lb) { return (kRecHeader + 3 * etab_size(la, lb) + 1) & ~1; }

// Compile-time loop: f(Ic<I>) for I = 0..N-1 (Ic<I> converts to the constant I).
template <int I>
struct Ic {
  static constexpr int value = I;
  constexpr __host__ __device__ operator int() const { return I; }
};
template <typename F, int... I>
__device__ __forceinline__ void sfor_impl(F&& f, std::integer_sequence<int, I...>) {
  (f(Ic<I>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void sfor(F&& f) {
  if constexpr (N > 0) sfor_impl(f, std::make_integer_sequence<int, N>{});
}

// Per-thread array of N doubles: in registers (SH = false), or one column of a
// block-wide shared-memory table (element i of thread t at p[i * kXsBlock]).
// (Single-warp blocks pack the shared memory more tightly but measured slower
// on [pp|pp] (-5 %) and no faster on the exchange, gradient and 3-center runs.)
constexpr int kXsBlock = 64;
constexpr int kRegMaxDevices = 64;
template <bool SH, int N>
struct TArr {
  double r[N];
  __device__ __forceinline__ double& operator[](int i) { return r[i]; }
};
template <int N>
struct TArr<true, N> {
  double* p;
  __device__ __forceinline__ double& operator[](int i) { return p[i * kXsBlock]; }
};

// One step of Eq. r along an axis: X r1 + (i - 1) r2 for an entry of index i (no second term for i = 1, whose
// index would be -1; one FMA for i = 2).
template <int I, typename F>
__device__ __forceinline__ double raise(double X, double r1, F&& r2) {
  if constexpr (I == 1) return X * r1;
  else if constexpr (I == 2) return fma(X, r1, r2());
  else return fma((double)(I - 1), r2(), X * r1);
}
// Product ex ey ez of three E-table entries of blocks with nx, ny, nz Hermite terms: the (0, 0) block of a
// table is the number 1 and costs no multiplication (12 of the 60 FP64 instructions that [..|ps] had issued
// per primitive quartet).
template <int NX, int NY, int NZ>
__device__ __forceinline__ double eprod(const double* ex, const double* ey, const double* ez) {
  if constexpr (NX * NY * NZ == 1) return 1.0;
  else if constexpr (NX * NY == 1) return __ldg(ez);
  else if constexpr (NX * NZ == 1) return __ldg(ey);
  else if constexpr (NY * NZ == 1) return __ldg(ex);
  else if constexpr (NZ == 1) return __ldg(ex) * __ldg(ey);
  else if constexpr (NY == 1) return __ldg(ex) * __ldg(ez);
  else if constexpr (NX == 1) return __ldg(ey) * __ldg(ez);
  else return __ldg(ex) * __ldg(ey) * __ldg(ez);
}

// ---- contracted ket pairs [ps), [ds), [pp): sums of scaled R tables instead of one ket transform per primitive
// With s = zeta_d / zeta_q, r = 1 / (2 zeta_q) and X = C - D of the pair, Q - C = -s X and Q - D = (1 - s) X, and every
// Hermite coefficient E^cd_q of Eqs. E2rr1/E2rr2 is a polynomial in X with coefficients s^M (1-s)^N r^w, where q
// of total order T takes w = T + (l_c + l_d - M - N - T) / 2. X is the same for all primitives of the pair, so
//   [p|cd] = sum over (M, N, T), |q| = T of  c X^(M+N) S_MNT[p + q],   S_MNT[h] = sum_k (s^M (1-s)^N r^w)_k R_k[h],
// and a primitive quartet costs the accumulation of the S tables (orders T .. L_b + T of R) in place of the whole ket
// transform; the expansion runs once per bra primitive. FP64 instructions per primitive quartet: [fs|ps] 120 -> 54,
// [dp|pp] 660 -> 160 (of about 360 and 870 with R and the Boys seeds). The E tables' cancellations are the same ones
// (Q - C and Q - D enter as products of s with one distance, as accurate as the tables' own differences).
template <int LC, int LD>
struct KetSets {
  static constexpr int n = 0, M[1] = {}, N[1] = {}, T[1] = {};
};
template <>
struct KetSets<1, 0> {
  static constexpr int n = 2, M[2] = {1, 0}, N[2] = {0, 0}, T[2] = {0, 1};
};
template <>
struct KetSets<2, 0> {
  static constexpr int n = 4, M[4] = {2, 0, 1, 0}, N[4] = {0, 0, 0, 0}, T[4] = {0, 0, 1, 2};
};
template <>
struct KetSets<1, 1> {
  static constexpr int n = 5, M[5] = {1, 0, 1, 0, 0}, N[5] = {1, 0, 0, 1, 0}, T[5] = {0, 0, 1, 1, 2};
};
// one term of [p|cd]: coef * monomial(X) * S_set[p + q]; monomials 1, X, Y, Z, XX, XY, XZ, YY, YZ, ZZ
struct KetTerm {
  int cd, set, q[3], mono, coef;
};
constexpr __host__ __device__ int binom(int n, int k) { return k == 0 || k == n ? 1 : binom(n - 1, k - 1) + binom(n - 1, k); }
// ways in which k Gaussian coordinates become t Hermite indices and (k - t) / 2 contracted pairs
constexpr __host__ __device__ int hermite_ways(int k, int t) {
  int f = binom(k, t);
  for (int i = k - t - 1; i > 1; i -= 2) f *= i;
  return f;
}
constexpr __host__ __device__ int monomial(int x, int y, int z) {
  if (x + y + z == 0) return 0;
  if (x + y + z == 1) return x ? 1 : (y ? 2 : 3);
  return x == 2 ? 4 : (x == 1 ? (y ? 5 : 6) : (y == 2 ? 7 : (y == 1 ? 8 : 9)));
}
constexpr int kKetTermsMax = 39;
struct KetTermTable {
  KetTerm t[kKetTermsMax];
  int n;
};
template <int LC, int LD>
constexpr __host__ __device__ KetTermTable ket_terms() {
  KetTermTable r{};
  using S = KetSets<LC, LD>;
  for (int c = 0; c < ncart(LC); ++c)
    for (int d = 0; d < ncart(LD); ++d)
      for (int i = 0; i < S::n; ++i) {
        const int C[3] = {cx(LC, c), cy(LC, c), cz(LC, c)}, D[3] = {cx(LD, d), cy(LD, d), cz(LD, d)};
        // per axis: m of the c coordinates give Q - C, n of the d ones Q - D, t Hermite indices
        for (int m0 = 0; m0 <= C[0]; ++m0) for (int m1 = 0; m1 <= C[1]; ++m1) for (int m2 = 0; m2 <= C[2]; ++m2)
        for (int n0 = 0; n0 <= D[0]; ++n0) for (int n1 = 0; n1 <= D[1]; ++n1) for (int n2 = 0; n2 <= D[2]; ++n2)
        for (int t0 = 0; t0 <= 2; ++t0) for (int t1 = 0; t1 <= 2; ++t1) for (int t2 = 0; t2 <= 2; ++t2) {
          if (m0 + m1 + m2 != S::M[i] || n0 + n1 + n2 != S::N[i] || t0 + t1 + t2 != S::T[i]) continue;
          const int k0 = C[0] - m0 + D[0] - n0, k1 = C[1] - m1 + D[1] - n1, k2 = C[2] - m2 + D[2] - n2;
          if (k0 < t0 || k1 < t1 || k2 < t2 || ((k0 - t0) & 1) || ((k1 - t1) & 1) || ((k2 - t2) & 1)) continue;
          int f = binom(C[0], m0) * binom(C[1], m1) * binom(C[2], m2) * binom(D[0], n0) * binom(D[1], n1) *
                  binom(D[2], n2) * hermite_ways(k0, t0) * hermite_ways(k1, t1) * hermite_ways(k2, t2);
          if ((S::M[i] + S::T[i]) & 1) f = -f;   // Q - C = -s X, and the ket sign (-1)^|q| of Eq. pq
          r.t[r.n] = KetTerm{c * ncart(LD) + d, i, {t0, t1, t2}, monomial(m0 + n0, m1 + n1, m2 + n2), f};
          ++r.n;
        }
      }
  return r;
}
template <int LC, int LD>
struct KetTerms {
  static constexpr KetTermTable v = ket_terms<LC, LD>();
};
// S tables of a class: set i holds the orders T .. L_b + T at set_off(i); the sets of the first group go through
// registers when the tables are expanded, the second group lies behind [p|cd] (see k_reg)
template <int LA, int LB, int LC, int LD>
struct KetPlan {
  using S = KetSets<LC, LD>;
  static constexpr int Lb = LA + LB, NX = nherm(Lb) * ncart(LC) * ncart(LD);
  static constexpr bool XS = !reg_eligible(LA, LB, LC, LD);
  static constexpr __host__ __device__ int set_size(int i) { return nherm(Lb + S::T[i]) - nherm(S::T[i] - 1); }
  static constexpr __host__ __device__ int total() {
    int s = 0;
    for (int i = 0; i < S::n; ++i) s += set_size(i);
    return s;
  }
  // beside R in registers, or in the shared-memory region of [p|cd] (in registers too they would leave half the
  // warps: [fs|ps] K = 1,6,3,6 2.16 ms from shared memory, 2.56 from registers)
  static constexpr bool in_regs = !XS;
  // first group: the sets of the highest T first, as many as 96 doubles hold (all of them in registers)
  static constexpr __host__ __device__ bool first(int i) {
    if (in_regs) return true;
    int used = 0;
    bool in = false;
    for (int k = S::n - 1; k >= 0; --k) {
      const bool fits = used + set_size(k) <= 96;
      if (fits) used += set_size(k);
      if (k == i) in = fits;
    }
    return in;
  }
  static constexpr __host__ __device__ int first_size() {
    int s = 0;
    for (int i = 0; i < S::n; ++i) s += first(i) ? set_size(i) : 0;
    return s;
  }
  static constexpr int second_at = NX > first_size() ? NX : first_size();
  static constexpr __host__ __device__ int set_off(int i) {
    int s = in_regs || first(i) ? 0 : second_at;
    for (int k = 0; k < i; ++k) s += first(k) == first(i) ? set_size(k) : 0;
    return s;
  }
  // doubles per thread of the shared [p|cd] region, without and with the S tables
  static constexpr int plain = XS ? NX : 0;
  static constexpr int region = XS ? (in_regs ? NX : second_at + total() - first_size()) : 0;
};
// position of (t, u, v), T <= t + u + v <= N, in the [t][u][v] simplex of order N without its orders below T <= 2
constexpr __host__ __device__ int sidx(int N, int T, int t, int u, int v) {
  return hidx(N, t, u, v) - (T == 0 ? 0 : (T == 1 ? 1 : 2 + (t + u >= 1) + (t >= 1)));
}
// 64-thread blocks of an SM by shared memory (doubles per thread)
constexpr int xs_blocks(int doubles) { return 227 * 1024 / (doubles * kXsBlock * 8 + 1024); }
// Classes that use the S tables: those that keep their blocks per SM, or nearly so ([ds|ds] 7 -> 6 blocks: 1.27 -> 1.18
// ms); where the bigger region halves them ([dp|pp] store) the two forms take the same time. Not the [ds) kets of a
// bra of total order 4 (205 doubles), whose expansion does not fit the registers
template <int LA, int LB, int LC, int LD, bool DIGEST>
constexpr bool ket_sums_eligible() {
  if constexpr (KetSets<LC, LD>::n == 0) return false;
  else {
    using P = KetPlan<LA, LB, LC, LD>;
    if (!P::XS) return true;
    const int v = DIGEST ? ncart(LA) * ncart(LB) * ncart(LC) * ncart(LD) : 0;
    return P::total() <= 170 && 4 * xs_blocks(P::region + v) >= 3 * xs_blocks(P::plain + v);
  }
}
// Blocks per SM that the registers are limited for: as many as the shared memory holds, up to what the kernel's
// tables need (the expansion's first group, or R, and 60 registers beside them)
template <int LA, int LB, int LC, int LD, bool DIGEST>
constexpr int ket_sums_blocks() {
  using P = KetPlan<LA, LB, LC, LD>;
  if (!P::XS) return 2;
  const int v = DIGEST ? ncart(LA) * ncart(LB) * ncart(LC) * ncart(LD) : 0;
  const int tab = P::first_size() > nherm(LA + LB + LC + LD) ? P::first_size() : nherm(LA + LB + LC + LD);
  const int by_regs = 65536 / kXsBlock / (2 * tab + 60), by_smem = xs_blocks(P::region + v);
  const int b = by_regs < by_smem ? by_regs : by_smem;
  return b < 4 ? 4 : b;
}
// ket primitives per lane from which the expansion is paid back
constexpr int kKetSumsMin = 3;

// Boys seeds of one primitive quartet and its Hermite integrals [tuv] of orders 0 .. L (Eqs. 0m, r) in R.
template <int L>
__device__ __forceinline__ void hermite_R(const double* __restrict__ boys, double zp, double zq, double PQx, double PQy,
                                          double PQz, double pref, double* R) {
  const double s = zp + zq;
  const double R2 = PQx * PQx + PQy * PQy + PQz * PQz;
  // Boys seeds G[m] = (-2 rho)^m pref F_m(T), m = 0..L (Eq. 0m), rho = zp zq / s, T = rho R^2, without a
  // branch between the table and the asymptotic form F_m(T) = Gamma(m+1/2) / (2 T^(m+1/2)):
  // with y = 1/sqrt(s) below T = 64 and y = 1/sqrt(zp zq R^2) above, and b = -2 zp zq y^2,
  //   G[m] = C y b^m f_m,  f_m = F_m(T) below and Gamma(m+1/2)/2 above,
  // and the table's last row holds the constants (T is 1 there, a grid point). The branch had cost a
  // quarter of the FP64 issue slots of [ps|ss] (warps whose quartets lie on both sides run both).
  // exp(-T) / (2 T F_m) is below 1e-20 from T = 64 on for m <= 6. With this, the one-term E tables and the
  // coefficient 1 of Eq. r (40,000 quartets): [ss|ss] K = 6,6,6,6 5.74 -> 4.09 ms, [ps|ss] K = 3,6,6,6
  // 4.22 -> 2.88 ms, [dp|ps] K = 1,3,3,6 1.55 -> 1.39 ms.
  const double zz2 = -2.0 * zp * zq;              // -2 zp zq
  const double c2 = zz2 * R2;                  // -2 zp zq R^2
  const int hc = __double2hiint(c2) & 0x7fffffff;
  const bool far = hc >= __double2hiint(s) + (7 << 20);   // 2 zp zq R^2 >= 128 s, by the exponents
  // zp zq R^2 = c2 / -2: sign off, exponent less one
  const double y = rsqrt(far ? __hiloint2double(hc - (1 << 20), __double2loint(c2)) : s);
  const double y2 = y * y;
  const double T2 = c2 * y2;                   // -2 T
  // nearest grid point of spacing 1/16: the low word of T + 1.5 2^48
  const double tm = fma(T2, -0.5, 422212465065984.0);
  const double nd = fma(T2, 0.5, tm - 422212465065984.0);   // T0 - T
  const int i = far ? kBoysNgrid - 1 : min(__double2loint(tm) & 0x7fffffff, kBoysNgrid - 1);
  const double2* row = reinterpret_cast<const double2*>(boys + (size_t)i * kBoysRow);
  double G[L + 1];
  {
    const double bm = zz2 * y2;
    double pw = pref * y;
    sfor<L + 1>([&](auto m) {
      const double2 c01 = __ldg(row + 4 * m), c23 = __ldg(row + 4 * m + 1);
      const double2 c45 = __ldg(row + 4 * m + 2), c67 = __ldg(row + 4 * m + 3);
      double f = fma(c67.y, nd, c67.x);
      f = fma(f, nd, c45.y);
      f = fma(f, nd, c45.x);
      f = fma(f, nd, c23.y);
      f = fma(f, nd, c23.x);
      f = fma(f, nd, c01.y);
      f = fma(f, nd, c01.x);
      G[m] = pw * f;
      if constexpr (m < L) pw *= bm;
    });
  }
  // R^(n)_tuv for n = L..0 in one array indexed in the order-L simplex:
  // level n overwrites orders N = L-n..1 from the top down (an entry reads
  // orders N-1 and N-2 of level n+1, not yet overwritten), then [000]
  R[0] = G[L];
  sfor<L>([&](auto k) {
    constexpr int n = L - 1 - k;
    sfor<L - n>([&](auto j) {
      constexpr int N = L - n - j;
      sfor<N + 1>([&](auto t) {
        sfor<N + 1 - t>([&](auto u) {
          constexpr int v = N - t - u;
          double val;
          if constexpr (v > 0) {
            val = raise<v>(PQz, R[hidx(L, t, u, v - 1)], [&] { return R[hidx(L, t, u, v - 2)]; });
          } else if constexpr (u > 0) {
            val = raise<u>(PQy, R[hidx(L, t, u - 1, 0)], [&] { return R[hidx(L, t, u - 2, 0)]; });
          } else {
            val = raise<t>(PQx, R[hidx(L, t - 1, 0, 0)], [&] { return R[hidx(L, t - 2, 0, 0)]; });
          }
          R[hidx(L, t, u, v)] = val;
        });
      });
    });
    R[0] = G[n];
  });
}

// XS = false: R, [p|cd] and the shellset in registers (classes with
// reg_eligible). XS = true: R in registers, [p|cd] and the shellset in shared
// memory (classes with reg_xs_eligible, total angular momentum <= 6).
// KS = true: contracted ket pairs by sums of scaled R tables (KetSets).
template <int LA, int LB, int LC, int LD, bool DIGEST, bool XS, bool KS>
__global__ void __launch_bounds__(XS ? kXsBlock : 128, KS ? ket_sums_blocks<LA, LB, LC, LD, DIGEST>() : 0) k_reg(const QuartetLaunch a) {
  constexpr int Lb = LA + LB, Lk = LC + LD, L = Lb + Lk;
  constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD);
  constexpr int Nb = NA * NB, Nk = NC * ND;
  constexpr int HB = nherm(Lb), HL = nherm(L);
  constexpr int RB = rec_size(LA, LB), RK = rec_size(LC, LD);
  constexpr int EB = etab_size(LA, LB), EK = etab_size(LC, LD);

  extern __shared__ double xs_smem[];
  // 2^(split_b + split_k) neighbouring lanes share a quartet: lane (sb, sk) takes the bra primitive pairs
  // sb, sb + Sb, ... and of each the ket primitive pairs sk, sk + Sk, ... (see split_of)
  const int lS = a.split_b + a.split_k, S = 1 << lS;
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t q = gid >> lS;
  if (q >= a.nq) return;   // whole lane groups leave together
  const int sub = (int)gid & (S - 1);
  const int Sb = 1 << a.split_b, Sk = 1 << a.split_k, sb = sub >> a.split_k, sk = sub & (Sk - 1);
  const unsigned grp = (S == 32 ? 0xffffffffu : (1u << S) - 1u) << (threadIdx.x & 31 & ~(S - 1));
  const int2 qp = a.qpairs[q];
  const double* __restrict__ rb0 = a.recs + a.pair_rec[qp.x + a.bra_var_off];
  const double* __restrict__ rk0 = a.recs_signed + a.pair_rec[qp.y + a.ket_var_off];
  const double* __restrict__ boys = a.boys;
  const int Kb = a.plan.Kb, Kk = a.plan.Kk;

  // shared-memory variant: [p|cd] in shared memory, and the shellset too when the digestion epilogue needs
  // it whole; the store epilogue adds each bra pair's row straight into the output instead (less shared
  // memory per thread, more warps per SM)
  constexpr bool VSH = XS && DIGEST;
  TArr<XS, Nb * Nk> V;
  TArr<XS, HB * Nk> X;
  if constexpr (XS) {
    V.p = xs_smem + (threadIdx.x & ~(S - 1));   // the shellset column of the group's first lane
    X.p = xs_smem + (VSH ? Nb * Nk : 0) * kXsBlock + threadIdx.x;
  }
  if constexpr (!XS) sfor<Nb * Nk>([&](auto i) { V[i] = 0.0; });
  // KS: the S tables in registers or, before [p|cd] takes their place, in its shared-memory region; monomials of C - D
  using KP = KetPlan<LA, LB, LC, LD>;
  constexpr bool SSH = KS && !KP::in_regs;
  constexpr int NS = KS ? KP::total() : 1;
  TArr<SSH, NS> SR;
  double mono[KS ? 10 : 1];
  if constexpr (KS) {
    if constexpr (SSH) SR.p = X.p;
    const double* E10 = rk0 + kRecHeader + etab_off(LD, 1, 0);
    if constexpr (LD > 0) {
      const double* E01 = rk0 + kRecHeader + etab_off(LD, 0, 1);
      sfor<3>([&](auto x) { mono[1 + x] = __ldg(E01 + x * EK) - __ldg(E10 + x * EK); });   // (Q - D) - (Q - C)
    } else {
      // from the primitive with the largest |s|: the error of X times any s is at most that of Q - C itself.
      // (Q - C below 1e-140 X is nothing beside 1 / zeta_q's terms; dividing its rounding by such an s would give an X
      // whose square is infinite)
      int top = -1, at = 0;
      for (int k = 0; k < Kk; ++k) {
        const int h = __double2hiint(__ldg(rk0 + (int64_t)k * RK + 7)) & 0x7fffffff;
        if (h > top) { top = h; at = k; }
      }
      const double sm = __ldg(rk0 + (int64_t)at * RK + 7);
      const double is = fabs(sm) > 1e-140 ? -1.0 / sm : 0.0;
      sfor<3>([&](auto x) { mono[1 + x] = __ldg(E10 + (int64_t)at * RK + x * EK) * is; });
    }
    mono[0] = 1.0;
    if constexpr (Lk > 1) {
      mono[4] = mono[1] * mono[1]; mono[5] = mono[1] * mono[2]; mono[6] = mono[1] * mono[3];
      mono[7] = mono[2] * mono[2]; mono[8] = mono[2] * mono[3]; mono[9] = mono[3] * mono[3];
    }
  }
  double* const outq = DIGEST ? nullptr : a.out + (a.qout ? a.qout[q] : q * (int64_t)(Nb * Nk));

  for (int pb0 = 0; pb0 < Kb; pb0 += Sb) {
    const bool live = pb0 + sb < Kb;   // a lane past the last bra primitive adds zeros to the group's sums
    const int pb = live ? pb0 + sb : 0;
    const double* __restrict__ rb = rb0 + (int64_t)pb * RB;
    const double zp = __ldg(rb);
    const double Px = __ldg(rb + 2), Py = __ldg(rb + 3), Pz = __ldg(rb + 4);
    // 2 pi^(5/2) * c_a c_b K_ab / zp (the ket part and 1/sqrt(zp+zq) per ket primitive)
    const double prefb = 34.986836655249725693 * __ldg(rb + 6);
    if constexpr (KS) {
      sfor<KetSets<LC, LD>::n>([&](auto i) {
        sfor<KP::set_size(i)>([&](auto h) { SR[KP::set_off(i) + h] = 0.0; });
      });
    } else {
      sfor<HB * Nk>([&](auto i) { X[i] = 0.0; });
    }

    for (int pk = live ? sk : Kk; pk < Kk; pk += Sk) {
      const double* __restrict__ rk = rk0 + (int64_t)pk * RK;
      const double zq = __ldg(rk);
      const double PQx = Px - __ldg(rk + 2), PQy = Py - __ldg(rk + 3), PQz = Pz - __ldg(rk + 4);
      double R[HL];
      hermite_R<L>(boys, zp, zq, PQx, PQy, PQz, prefb * __ldg(rk + 6), R);
      if constexpr (KS) {
        using S = KetSets<LC, LD>;
        const double zs = __ldg(rk + 7), zr = -__ldg(rk + kRecHeader + etab_off(LD, 1, 0) + 1);   // signed table: -r
        sfor<S::n>([&](auto i) {
          constexpr int M1 = S::M[i], N1 = S::N[i], T1 = S::T[i];
          constexpr int w = T1 + (Lk - M1 - N1 - T1) / 2, N = Lb + T1;
          double f = 1.0;
          if constexpr (N1 > 0) f = 1.0 - zs;
          else if constexpr (M1 > 0) f = zs;
          if constexpr (M1 + N1 > 1) f *= zs;
          if constexpr (M1 + N1 > 0 && w > 0) f *= zr;
          else if constexpr (w > 0) f = zr;
          if constexpr (w > 1) f *= zr;
          sfor<N + 1>([&](auto t) {
            sfor<N + 1 - t>([&](auto u) {
              sfor<N + 1 - t - u>([&](auto v) {
                if constexpr (t + u + v >= T1) {
                  constexpr int o = KP::set_off(i) + sidx(N, T1, t, u, v);
                  SR[o] = fma(f, R[hidx(L, t, u, v)], SR[o]);
                }
              });
            });
          });
        });
      } else
      // ket transform: X[p][cd] += sum_{tau,nu,phi} Ex Ey Ez (signed tables) R[p + q]
      sfor<NC>([&](auto c) {
        sfor<ND>([&](auto d) {
          constexpr int ex = cx(LC, c), ey = cy(LC, c), ez = cz(LC, c);
          constexpr int fx = cx(LD, d), fy = cy(LD, d), fz = cz(LD, d);
          constexpr int nx = ex + fx + 1, ny = ey + fy + 1, nz = ez + fz + 1;
          const double* Ex = rk + kRecHeader + etab_off(LD, ex, fx);
          const double* Ey = rk + kRecHeader + EK + etab_off(LD, ey, fy);
          const double* Ez = rk + kRecHeader + 2 * EK + etab_off(LD, ez, fz);
          double E[nx * ny * nz];
          sfor<nx * ny * nz>([&](auto k) {
            E[k] = eprod<nx, ny, nz>(Ex + k / (ny * nz), Ey + k / nz % ny, Ez + k % nz);
          });
          sfor<Lb + 1>([&](auto t) {
            sfor<Lb + 1 - t>([&](auto u) {
              sfor<Lb + 1 - t - u>([&](auto v) {
                constexpr int o = hidx(Lb, t, u, v) * Nk + c * ND + d;
                double acc = X[o];
                sfor<nx>([&](auto tau) {
                  sfor<ny>([&](auto nu) {
                    sfor<nz>([&](auto phi) {
                      const double r = R[hidx(L, t + tau, u + nu, v + phi)];
                      if constexpr (nx * ny * nz == 1) acc += r;
                      else acc = fma(E[(tau * ny + nu) * nz + phi], r, acc);
                    });
                  });
                });
                X[o] = acc;
              });
            });
          });
        });
      });
    }
    if constexpr (KS) {
      // [p|cd] from the S tables: those of the first group pass through registers, since [p|cd] takes their place
      using KT = KetTerms<LC, LD>;
      constexpr int NF = KP::first_size(), second = NS - NF;
      double F[SSH ? NF : 1];
      if constexpr (SSH) sfor<NF>([&](auto i) { F[i] = SR[i]; });
      auto expand = [&](auto grp2) {   // the terms of one group; the second adds to the first
        sfor<Lb + 1>([&](auto t) {
          sfor<Lb + 1 - t>([&](auto u) {
            sfor<Lb + 1 - t - u>([&](auto v) {
              constexpr int h = hidx(Lb, t, u, v) * Nk;
              double x[Nk];
              sfor<Nk>([&](auto cd) { x[cd] = grp2 ? X[h + cd] : 0.0; });
              sfor<KT::v.n>([&](auto k) {
                constexpr KetTerm e = KT::v.t[k];
                if constexpr (KP::first(e.set) != (grp2 == 1)) {
                  constexpr int T = KetSets<LC, LD>::T[e.set];
                  constexpr int o = KP::set_off(e.set) + sidx(Lb + T, T, t + e.q[0], u + e.q[1], v + e.q[2]);
                  double y;
                  if constexpr (SSH && !(grp2 == 1)) y = F[o];
                  else y = SR[o];
                  if constexpr (e.mono == 0 && e.coef == 1) x[e.cd] += y;
                  else if constexpr (e.mono == 0 && e.coef == -1) x[e.cd] -= y;
                  else x[e.cd] = fma((double)e.coef * mono[e.mono], y, x[e.cd]);
                }
              });
              sfor<Nk>([&](auto cd) { X[h + cd] = x[cd]; });
            });
          });
        });
      };
      expand(Ic<0>{});
      if constexpr (second > 0) expand(Ic<1>{});
    }
    // bra transform: V[ab][cd] += sum_{t,u,v} Ex Ey Ez X[tuv][cd]
    if constexpr (XS) {
      // [p|cd] and the shellset are in shared memory: runtime loops over ab and
      // (t,u,v), the ket pairs cd unrolled (keeps the unrolled body small)
      for (int ia = 0; ia < NA; ++ia) {
        const int ax = cx(LA, ia), ay = cy(LA, ia), az = LA - ax - ay;
        for (int ib = 0; ib < NB; ++ib) {
          const int bx = cx(LB, ib), by = cy(LB, ib), bz = LB - bx - by;
          const double* Ex = rb + kRecHeader + etab_off(LB, ax, bx);
          const double* Ey = rb + kRecHeader + EB + etab_off(LB, ay, by);
          const double* Ez = rb + kRecHeader + 2 * EB + etab_off(LB, az, bz);
          double acc[Nk];
          sfor<Nk>([&](auto cd) { acc[cd] = 0.0; });
          for (int t = 0; t <= ax + bx; ++t) {
            const double vx = __ldg(Ex + t);
            for (int u = 0; u <= ay + by; ++u) {
              // (a one-term table is the number 1; the uniform branch also makes the faster loop: [pp|pp] 161 -> 152 us)
              const double vxy = ay + by ? vx * __ldg(Ey + u) : vx;
              for (int v = 0; v <= az + bz; ++v) {
                const double e = az + bz ? vxy * __ldg(Ez + v) : vxy;
                const int h = hidx(Lb, t, u, v) * Nk;
                sfor<Nk>([&](auto cd) { acc[cd] = fma(e, X[h + cd], acc[cd]); });
              }
            }
          }
          const int o = (ia * NB + ib) * Nk;
          if (S == 1) {
            if constexpr (VSH) {
              if (pb0 == 0) sfor<Nk>([&](auto cd) { V[o + cd] = acc[cd]; });
              else sfor<Nk>([&](auto cd) { V[o + cd] += acc[cd]; });
            } else if (pb0 == 0) {
              sfor<Nk>([&](auto cd) { outq[o + cd] = acc[cd]; });
            } else {
              sfor<Nk>([&](auto cd) { outq[o + cd] += acc[cd]; });
            }
            continue;
          }
          for (int off = 1; off < S; off <<= 1)   // the group's sum, in every lane
            sfor<Nk>([&](auto cd) { acc[cd] += __shfl_xor_sync(grp, acc[cd], off); });
          sfor<Nk>([&](auto cd) {
            if ((cd & (S - 1)) != sub) return;   // the lanes of the group share the row's elements
            double* dst;
            if constexpr (VSH) dst = &V[o + cd];
            else dst = outq + o + cd;
            *dst = pb0 == 0 ? acc[cd] : *dst + acc[cd];
          });
        }
      }
    } else {
      sfor<NA>([&](auto ia) {
        sfor<NB>([&](auto ib) {
          constexpr int ax = cx(LA, ia), ay = cy(LA, ia), az = cz(LA, ia);
          constexpr int bx = cx(LB, ib), by = cy(LB, ib), bz = cz(LB, ib);
          constexpr int nx = ax + bx + 1, ny = ay + by + 1, nz = az + bz + 1;
          const double* Ex = rb + kRecHeader + etab_off(LB, ax, bx);
          const double* Ey = rb + kRecHeader + EB + etab_off(LB, ay, by);
          const double* Ez = rb + kRecHeader + 2 * EB + etab_off(LB, az, bz);
          double E[nx * ny * nz];
          sfor<nx * ny * nz>([&](auto k) {
            E[k] = eprod<nx, ny, nz>(Ex + k / (ny * nz), Ey + k / nz % ny, Ez + k % nz);
          });
          sfor<Nk>([&](auto cd) {
            constexpr int o = (ia * NB + ib) * Nk + cd;
            double acc = V[o];
            sfor<nx>([&](auto t) {
              sfor<ny>([&](auto u) {
                sfor<nz>([&](auto v) {
                  const double x = X[hidx(Lb, t, u, v) * Nk + cd];
                  if constexpr (nx * ny * nz == 1) acc += x;
                  else acc = fma(E[(t * ny + u) * nz + v], x, acc);
                });
              });
            });
            V[o] = acc;
          });
        });
      });
    }
  }

  if constexpr (!XS) {
    for (int off = 1; off < S; off <<= 1)
      sfor<Nb * Nk>([&](auto i) { V[i] += __shfl_xor_sync(grp, V[i], off); });
  }
  if constexpr (VSH) __syncwarp(grp);   // every lane reads the shellset below
  if constexpr (!DIGEST) {
    // (no offsets: shellsets back to back); the shared-memory variant has written its rows already
    if constexpr (!XS) {
      if (S == 1) sfor<Nb * Nk>([&](auto i) { outq[i] = V[i]; });
      else
        sfor<Nb * Nk>([&](auto i) {
          if ((i & (S - 1)) == sub) outq[i] = V[i];
        });
    }
  } else {
    // Exchange digestion of the unique quartet (ij|kl) with weight w, as in
    // the team kernel: K_ik += w D_jl V, K_il += w D_jk V, K_jk += w D_il V,
    // K_jl += w D_ik V (the host adds K^T afterwards).
    const int2 bp = a.pair_shells[qp.x], kp = a.pair_shells[qp.y];
    const int si = bp.x, sj = bp.y, sk = kp.x, sl = kp.y;
    const double w = (si == sj ? 0.5 : 1.0) * (sk == sl ? 0.5 : 1.0) * (qp.x == qp.y ? 0.5 : 1.0);
    const int mol = a.pair_mol ? a.pair_mol[qp.x] : -1;
    const int64_t nao = mol >= 0 ? a.mol_nao[mol] : a.nao;
    const double* __restrict__ D = mol >= 0 ? a.mol_D[mol] : a.D;
    double* K = mol >= 0 ? a.mol_K[mol] : a.K;
    const int64_t ai = a.ao_off[si], aj = a.ao_off[sj], ak = a.ao_off[sk], al = a.ao_off[sl];
    if constexpr (XS) {
      // the shellset is in shared memory: runtime loops
      auto Vr = [&](int x, int b, int c, int d) -> double { return V[((x * NB + b) * NC + c) * ND + d]; };
      for (int x = 0; x < NA; ++x) {
        for (int c = 0; c < NC; ++c) {   // K_ik
          if (((x * NC + c) & (S - 1)) != sub) continue;   // the group's lanes share the elements of each block
          double s1 = 0.0;
          for (int b = 0; b < NB; ++b)
            for (int d = 0; d < ND; ++d) s1 = fma(__ldg(D + (aj + b) * nao + al + d), Vr(x, b, c, d), s1);
          atomicAdd(K + (ai + x) * nao + ak + c, w * s1);
        }
        for (int d = 0; d < ND; ++d) {   // K_il
          if (((x * ND + d) & (S - 1)) != sub) continue;
          double s2 = 0.0;
          for (int b = 0; b < NB; ++b)
            for (int c = 0; c < NC; ++c) s2 = fma(__ldg(D + (aj + b) * nao + ak + c), Vr(x, b, c, d), s2);
          atomicAdd(K + (ai + x) * nao + al + d, w * s2);
        }
      }
      for (int x = 0; x < NB; ++x) {
        for (int c = 0; c < NC; ++c) {   // K_jk
          if (((x * NC + c) & (S - 1)) != sub) continue;
          double s3 = 0.0;
          for (int y = 0; y < NA; ++y)
            for (int d = 0; d < ND; ++d) s3 = fma(__ldg(D + (ai + y) * nao + al + d), Vr(y, x, c, d), s3);
          atomicAdd(K + (aj + x) * nao + ak + c, w * s3);
        }
        for (int d = 0; d < ND; ++d) {   // K_jl
          if (((x * ND + d) & (S - 1)) != sub) continue;
          double s4 = 0.0;
          for (int y = 0; y < NA; ++y)
            for (int c = 0; c < NC; ++c) s4 = fma(__ldg(D + (ai + y) * nao + ak + c), Vr(y, x, c, d), s4);
          atomicAdd(K + (aj + x) * nao + al + d, w * s4);
        }
      }
    } else {
      auto Vat = [&](auto x, auto b, auto c, auto d) -> double { return V[((x * NB + b) * NC + c) * ND + d]; };
      sfor<NA>([&](auto x) {
        sfor<NC>([&](auto c) {   // K_ik
          if (((x * NC + c) & (S - 1)) != sub) return;
          double s1 = 0.0;
          sfor<NB>([&](auto b) {
            sfor<ND>([&](auto d) { s1 = fma(__ldg(D + (aj + b) * nao + al + d), Vat(x, b, c, d), s1); });
          });
          atomicAdd(K + (ai + x) * nao + ak + c, w * s1);
        });
        sfor<ND>([&](auto d) {   // K_il
          if (((x * ND + d) & (S - 1)) != sub) return;
          double s2 = 0.0;
          sfor<NB>([&](auto b) {
            sfor<NC>([&](auto c) { s2 = fma(__ldg(D + (aj + b) * nao + ak + c), Vat(x, b, c, d), s2); });
          });
          atomicAdd(K + (ai + x) * nao + al + d, w * s2);
        });
      });
      sfor<NB>([&](auto x) {
        sfor<NC>([&](auto c) {   // K_jk
          if (((x * NC + c) & (S - 1)) != sub) return;
          double s3 = 0.0;
          sfor<NA>([&](auto y) {
            sfor<ND>([&](auto d) { s3 = fma(__ldg(D + (ai + y) * nao + al + d), Vat(y, x, c, d), s3); });
          });
          atomicAdd(K + (aj + x) * nao + ak + c, w * s3);
        });
        sfor<ND>([&](auto d) {   // K_jl
          if (((x * ND + d) & (S - 1)) != sub) return;
          double s4 = 0.0;
          sfor<NA>([&](auto y) {
            sfor<NC>([&](auto c) { s4 = fma(__ldg(D + (ai + y) * nao + ak + c), Vat(y, x, c, d), s4); });
          });
          atomicAdd(K + (aj + x) * nao + al + d, w * s4);
        });
      });
    }
  }
}

// How many lanes share a quartet (log2, over the bra and the ket primitive pairs). A launch of few quartets
// of a contracted class is bound by the chain of primitive quartets that one thread runs (1.8 us each for
// [ss|ss]), not by the FP64 pipe: its time is taken as the chain's work, times the number of times the
// launch's lanes exceed kSatThreads, from where on the pipe is busy and lanes that idle in a partial round
// of primitives cost as much as working ones. Measured: one-shot 4-center call on 2 atoms 77.1 -> 23.0 ms,
// on 6 atoms 87.5 -> 26.0 ms, density fitting of 4 atoms 11.8 -> 6.1 ms, 8-molecule batched exchange
// 163 -> 113 ms; launches of more than 24,000 quartets keep one lane each and their time. ck / cb: FP64 operations per primitive quartet and per bra
// transform; cr: per step of the lanes' reduction.
constexpr double kSatThreads = 152 * 160.0;
inline void split_of(int64_t nq, int concurrent, int Kb, int Kk, double ck, double cb, double cr, int* lb, int* lk) {
  const double sat = kSatThreads / std::max(1, concurrent);   // this launch's share of the SMs
  double best = 1e300;
  *lb = *lk = 0;
  for (int ls = 0; ls <= 5; ++ls)
    for (int b = 0; b <= ls; ++b) {
      const int k = ls - b;
      if ((b && (1 << b) >= 2 * Kb) || (k && (1 << k) >= 2 * Kk)) continue;
      const double rounds = (Kb + (1 << b) - 1) >> b, per = (Kk + (1 << k) - 1) >> k;
      const double chain = rounds * (per * ck + cb) + ls * cr;
      const double t = chain * std::max(1.0, (double)nq * (1 << ls) / sat);
      if (t < 0.97 * best) { best = t; *lb = b; *lk = k; }
    }
}

// The cost arguments of split_of for a class.
struct SplitCost {
  double ck, cb, cr;
};
constexpr SplitCost split_cost(int la, int lb, int lc, int ld) {
  const double body = reg_body_size(la, lb, lc, ld), ket = reg_body_size(la, lb, lc, ld, false);
  return {ket + 8.0 * (la + lb + lc + ld + 1) + 80.0, body - ket,
          (double)(ncart(la) * ncart(lb) * ncart(lc) * ncart(ld))};
}
// Ket primitives per lane decide between the instance that sums R tables and the one that does not.
inline bool runs_sums(int Kk, int split_k) { return ((Kk + (1 << split_k) - 1) >> split_k) >= kKetSumsMin; }

// Uncontracted shellsets of the classes below: one warp per block, one thread per quartet, everything in registers. The
// columns [p|cd] are formed one at a time and go through the bra transform at once, so that neither [p|cd] nor the
// shellset is ever whole; the products of the bra's E tables are formed once. The shared-memory variant holds [p|cd]
// of a class ([pp|pp]: 46 KB per 64 threads, 8 warps per SM), which made 1.3 waves of the sweep's 50,176 quartets and
// kept the FP64 pipe 51 % busy; here 12 warps fit and the launch is one wave. 50,176 quartets: [pp|pp] 151 -> 103 us,
// [ds|pp] 122 -> 91, [sp|sg] 130 -> 116; 100 quartets: 62 -> 48, 54 -> 44, 58 -> 54 us (pair records included).
template <int LA, int LB>
struct BraTerms {   // Hermite terms of the Cartesian bra pairs, pair by pair
  static constexpr __host__ __device__ int size(int ia, int ib) {
    return (cx(LA, ia) + cx(LB, ib) + 1) * (cy(LA, ia) + cy(LB, ib) + 1) * (cz(LA, ia) + cz(LB, ib) + 1);
  }
  static constexpr __host__ __device__ int off(int ia, int ib) {
    int s = 0;
    for (int k = 0; k < ia * ncart(LB) + ib; ++k) s += size(k / ncart(LB), k % ncart(LB));
    return s;
  }
  static constexpr __host__ __device__ int total() { return off(ncart(LA), 0); }
};
// R and the bra products within 72 doubles, and a body that compiles quickly
template <int LA, int LB, int LC, int LD>
constexpr bool single_eligible() {
  return !reg_eligible(LA, LB, LC, LD) && nherm(LA + LB + LC + LD) + BraTerms<LA, LB>::total() <= 72 &&
         reg_body_size(LA, LB, LC, LD) <= 1000;
}
template <int LA, int LB, int LC, int LD>
__global__ void __launch_bounds__(32, 12) k_reg_single(const QuartetLaunch a) {
  constexpr int Lb = LA + LB, L = Lb + LC + LD;
  constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD), Nk = NC * ND;
  constexpr int EB = etab_size(LA, LB), EK = etab_size(LC, LD);
  using BT = BraTerms<LA, LB>;
  const int64_t q = (int64_t)blockIdx.x * 32 + threadIdx.x;
  if (q >= a.nq) return;
  const int2 qp = a.qpairs[q];
  const double* __restrict__ rb = a.recs + a.pair_rec[qp.x + a.bra_var_off];
  const double* __restrict__ rk = a.recs_signed + a.pair_rec[qp.y + a.ket_var_off];
  double* const outq = a.out + (a.qout ? a.qout[q] : q * (int64_t)(NA * NB * Nk));
  double R[nherm(L)];
  hermite_R<L>(a.boys, __ldg(rb), __ldg(rk), __ldg(rb + 2) - __ldg(rk + 2), __ldg(rb + 3) - __ldg(rk + 3),
               __ldg(rb + 4) - __ldg(rk + 4), 34.986836655249725693 * __ldg(rb + 6) * __ldg(rk + 6), R);
  double B[BT::total()];
  sfor<NA>([&](auto ia) {
    sfor<NB>([&](auto ib) {
      constexpr int ax = cx(LA, ia), ay = cy(LA, ia), az = cz(LA, ia);
      constexpr int bx = cx(LB, ib), by = cy(LB, ib), bz = cz(LB, ib);
      constexpr int nx = ax + bx + 1, ny = ay + by + 1, nz = az + bz + 1, o = BT::off(ia, ib);
      const double* Ex = rb + kRecHeader + etab_off(LB, ax, bx);
      const double* Ey = rb + kRecHeader + EB + etab_off(LB, ay, by);
      const double* Ez = rb + kRecHeader + 2 * EB + etab_off(LB, az, bz);
      sfor<nx * ny * nz>([&](auto k) {
        B[o + k] = eprod<nx, ny, nz>(Ex + k / (ny * nz), Ey + k / nz % ny, Ez + k % nz);
      });
    });
  });
  sfor<NC>([&](auto c) {
    sfor<ND>([&](auto d) {
      double X[nherm(Lb)];
      {
        constexpr int ex = cx(LC, c), ey = cy(LC, c), ez = cz(LC, c);
        constexpr int fx = cx(LD, d), fy = cy(LD, d), fz = cz(LD, d);
        constexpr int nx = ex + fx + 1, ny = ey + fy + 1, nz = ez + fz + 1;
        const double* Ex = rk + kRecHeader + etab_off(LD, ex, fx);
        const double* Ey = rk + kRecHeader + EK + etab_off(LD, ey, fy);
        const double* Ez = rk + kRecHeader + 2 * EK + etab_off(LD, ez, fz);
        double E[nx * ny * nz];
        sfor<nx * ny * nz>([&](auto k) {
          E[k] = eprod<nx, ny, nz>(Ex + k / (ny * nz), Ey + k / nz % ny, Ez + k % nz);
        });
        sfor<Lb + 1>([&](auto t) {
          sfor<Lb + 1 - t>([&](auto u) {
            sfor<Lb + 1 - t - u>([&](auto v) {
              double acc = 0.0;
              sfor<nx * ny * nz>([&](auto k) {
                const double r = R[hidx(L, t + k / (ny * nz), u + k / nz % ny, v + k % nz)];
                if constexpr (nx * ny * nz == 1) acc = r;
                else if constexpr (k == 0) acc = E[k] * r;
                else acc = fma(E[k], r, acc);
              });
              X[hidx(Lb, t, u, v)] = acc;
            });
          });
        });
      }
      sfor<NA>([&](auto ia) {
        sfor<NB>([&](auto ib) {
          constexpr int ny = cy(LA, ia) + cy(LB, ib) + 1, nz = cz(LA, ia) + cz(LB, ib) + 1, n = BT::size(ia, ib), o = BT::off(ia, ib);
          double acc = 0.0;
          sfor<n>([&](auto k) {
            const double x = X[hidx(Lb, k / (ny * nz), k / nz % ny, k % nz)];
            if constexpr (n == 1) acc = x;
            else if constexpr (k == 0) acc = B[o] * x;
            else acc = fma(B[o + k], x, acc);
          });
          outq[(ia * NB + ib) * Nk + c * ND + d] = acc;
        });
      });
    });
  });
}

// The instance of one epilogue: with the S tables of the ket pair where the class has them and each lane runs
// enough ket primitives.
template <int LA, int LB, int LC, int LD, bool DIGEST>
cudaError_t launch_reg_epilogue(const QuartetLaunch& a, unsigned grid, cudaStream_t s) {
  constexpr bool XS = !reg_eligible(LA, LB, LC, LD);
  constexpr int bs = XS ? kXsBlock : 128;
  // shared memory per block: [p|cd] or the S tables (and, with the digestion epilogue, the shellset) of every thread
  using P = KetPlan<LA, LB, LC, LD>;
  constexpr int v = XS && DIGEST ? ncart(LA) * ncart(LB) * ncart(LC) * ncart(LD) : 0;
  constexpr size_t shm = (size_t)(P::plain + v) * kXsBlock * sizeof(double);
  constexpr bool KS = ket_sums_eligible<LA, LB, LC, LD, DIGEST>();
  constexpr size_t shm_s = KS ? (size_t)(P::region + v) * kXsBlock * sizeof(double) : shm;
  auto* const plain = k_reg<LA, LB, LC, LD, DIGEST, XS, false>;
  auto* const sums = k_reg<LA, LB, LC, LD, DIGEST, XS, KS>;
  if constexpr (shm_s > 48 * 1024) {
    // opt in to more than 48 KB of dynamic shared memory, once per instance and device
    static bool attr[kRegMaxDevices] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kRegMaxDevices) return cudaErrorInvalidDevice;
    if (!attr[dev]) {
      e = cudaFuncSetAttribute(plain, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(sums, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm_s);
      if (e != cudaSuccess) return e;
      attr[dev] = true;
    }
  }
  if constexpr (!DIGEST && single_eligible<LA, LB, LC, LD>()) {
    if (a.plan.Kb * a.plan.Kk == 1) {
      k_reg_single<LA, LB, LC, LD><<<(unsigned)((a.nq + 31) / 32), 32, 0, s>>>(a);
      return cudaGetLastError();
    }
  }
  if (KS && runs_sums(a.plan.Kk, a.split_k)) sums<<<grid, bs, shm_s, s>>>(a);
  else plain<<<grid, bs, shm, s>>>(a);
  return cudaGetLastError();
}

template <int LA, int LB, int LC, int LD>
cudaError_t launch_reg_class(const QuartetLaunch& a0, cudaStream_t s) {
  constexpr bool XS = !reg_eligible(LA, LB, LC, LD);
  constexpr int bs = XS ? kXsBlock : 128;
  QuartetLaunch a = a0;
  constexpr SplitCost sc = split_cost(LA, LB, LC, LD);
  split_of(a.share_nq ? a.share_nq : a.nq, a.concurrent, a.plan.Kb, a.plan.Kk, sc.ck, sc.cb, sc.cr, &a.split_b,
           &a.split_k);
  const int64_t grid = ((a.nq << (a.split_b + a.split_k)) + bs - 1) / bs;
  if (grid > 0x7fffffff) return cudaErrorInvalidValue;
  return a.D ? launch_reg_epilogue<LA, LB, LC, LD, true>(a, (unsigned)grid, s)
             : launch_reg_epilogue<LA, LB, LC, LD, false>(a, (unsigned)grid, s);
}

using RegLaunchFn = cudaError_t (*)(const QuartetLaunch&, cudaStream_t);

// Launcher of class code C = ((la*7 + lb)*7 + lc)*7 + ld, or nullptr when the
// class has no register kernel.
template <int C>
constexpr RegLaunchFn reg_fn() {
  constexpr int la = C / 343, lb = C / 49 % 7, lc = C / 7 % 7, ld = C % 7;
  if constexpr (reg_eligible(la, lb, lc, ld) || reg_xs_eligible(la, lb, lc, ld))
    return &launch_reg_class<la, lb, lc, ld>;
  else return nullptr;
}
template <int BASE, int... I>
__host__ RegLaunchFn reg_pick(int code, std::integer_sequence<int, I...>) {
  constexpr RegLaunchFn table[] = {reg_fn<BASE + I>()...};
  return table[code - BASE];
}

}  // namespace reg
}  // namespace mdx
