// What a register-kernel launch chooses (reg_kernel.cuh) and the work it then does, for reports.
#include "reg_kernel.cuh"

namespace mdx {
namespace reg {
namespace {

// A class's instances: whether the sums of scaled R tables exist for the store and the digestion epilogue, their FP64
// instructions per primitive quartet (in place of the ket transform) and per bra primitive, and whether k_reg_single
// takes its uncontracted shellsets.
struct ClassInfo {
  bool sums_store = false, sums_digest = false, single = false;
  int per_prim = 0, per_bra = 0;
};
template <int LA, int LB, int LC, int LD>
constexpr ClassInfo class_info() {
  ClassInfo r;
  r.single = single_eligible<LA, LB, LC, LD>();
  r.sums_store = ket_sums_eligible<LA, LB, LC, LD, false>();
  r.sums_digest = ket_sums_eligible<LA, LB, LC, LD, true>();
  if constexpr (KetSets<LC, LD>::n > 0) {
    using S = KetSets<LC, LD>;
    r.per_prim = KetPlan<LA, LB, LC, LD>::total();
    for (int i = 0; i < S::n; ++i) {   // products of the factor s^M (1-s)^N r^w
      const int mn = S::M[i] + S::N[i], w = S::T[i] + (LC + LD - mn - S::T[i]) / 2;
      r.per_prim += (S::N[i] > 0) + (mn > 1) + (mn > 0 && w > 0) + (w > 1);
    }
    r.per_bra = nherm(LA + LB) * KetTerms<LC, LD>::v.n;
  }
  return r;
}
template <int C>
constexpr ClassInfo code_info() {
  constexpr int la = C / 343, lb = C / 49 % 7, lc = C / 7 % 7, ld = C % 7;
  if constexpr (reg_eligible(la, lb, lc, ld) || reg_xs_eligible(la, lb, lc, ld)) return class_info<la, lb, lc, ld>();
  else return ClassInfo{};
}
template <int... C>
ClassInfo pick(int code, std::integer_sequence<int, C...>) {
  static constexpr ClassInfo table[] = {code_info<C>()...};
  return table[code];
}

}  // namespace
}  // namespace reg

RegShape reg_shape(const PlanDev& P, int64_t nq, int concurrent, bool digest) {
  const reg::ClassInfo i = reg::pick(((P.la * 7 + P.lb) * 7 + P.lc) * 7 + P.ld, std::make_integer_sequence<int, 7 * 7 * 7 * 7>{});
  const reg::SplitCost c = reg::split_cost(P.la, P.lb, P.lc, P.ld);
  RegShape r{};
  reg::split_of(nq, concurrent, P.Kb, P.Kk, c.ck, c.cb, c.cr, &r.split_b, &r.split_k);
  r.single = !digest && i.single && P.Kb * P.Kk == 1;
  r.sums = !r.single && (digest ? i.sums_digest : i.sums_store) && reg::runs_sums(P.Kk, r.split_k);
  r.sums_per_prim = i.per_prim;
  r.sums_per_bra = i.per_bra;
  return r;
}

}  // namespace mdx
