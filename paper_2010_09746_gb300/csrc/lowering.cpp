// From a compiled pass's register ops to the ops the kernels run.
//
// The compiler's register ops are general: a phase table multiplies any subset of the register
// elements, a conditional phase names its slots by a mask.  Most of them depend on one or two
// slots only.  Those become ops whose slots are compile-time constants in the kernels (a dispatch
// on the slot, once per op): no mask test per element, one or three table entries loaded instead
// of one per element, and no products with entries that are exactly 1.  The arithmetic on every
// amplitude is unchanged.
//
// Measured: 25-qubit QFT complex128 (264 controlled phases, in groups of up to 12 on one slot)
// 9.01 -> 6.17 ms; 23-qubit Haar circuit complex128 16.4 -> 15.9 ms; complex64: 17 qubits
// 1163 -> 1117 us, 27-qubit RZ/RX/CZ 24.3 -> 23.7 ms, with the same bits.
#include <algorithm>

#include "qs_internal.h"

namespace qs {

namespace {

// the pattern of register indices with bit s set, over 2^K indices
uint32_t slot_pattern(int s, int K) {
  uint32_t m = 0;
  for (int j = 0; j < (1 << K); j++)
    if ((j >> s) & 1) m |= 1u << j;
  return m;
}

bool same_entry(const Pool& p, int a, int b) {
  return p.f64[2 * (size_t)a] == p.f64[2 * (size_t)b] && p.f64[2 * (size_t)a + 1] == p.f64[2 * (size_t)b + 1];
}

// a table whose entries depend on one or two slots only, with entry 1 where neither is set
void narrow_table(const Pool& pool, int K, RegOp* r) {
  if (r->csl == 0) {   // every entry is 1: nothing to do (a rotation run without slots)
    r->type = OP_RXTM;
    r->neg = 0;
    return;
  }
  for (int s = 0; s < K; s++)
    if (r->csl == slot_pattern(s, K)) {
      for (int j = 0; j < (1 << K); j++)
        if (((j >> s) & 1) && !same_entry(pool, r->mat + j, r->mat + (1 << s))) return;
      r->type = OP_PHASE;   // unconditional: multiply by entry 2^s where slot s is set
      r->s0 = (int8_t)s;
      r->mat += 1 << s;
      r->csl = 1u << s;
      r->neg = 0;
      return;
    }
  for (int a = 0; a < K; a++)
    for (int b = a + 1; b < K; b++)
      if (r->csl == (slot_pattern(a, K) | slot_pattern(b, K))) {
        for (int j = 0; j < (1 << K); j++) {
          const int e = j & ((1 << a) | (1 << b));
          if (e && !same_entry(pool, r->mat + j, r->mat + e)) return;
        }
        r->type = OP_DTAB2;
        r->s0 = (int8_t)a;
        r->s1 = (int8_t)b;
        return;
      }
}

}  // namespace

std::vector<RegOp> lower_regops(const CompileResult& cr) {
  std::vector<RegOp> ops = cr.reg_ops;
  for (const StageRec& st : cr.stages) {
    if (st.kind != 0) continue;
    const int K = __builtin_popcount((uint32_t)st.rmask);
    for (int i = st.op0; i < st.op0 + st.nops; i++) {
      RegOp& r = ops[i];
      if (r.type == OP_DTAB) narrow_table(cr.pool, K, &r);
      else if (r.type == OP_PHASE && __builtin_popcount(r.csl) == 1) r.s0 = (int8_t)__builtin_ctz(r.csl);
    }
    if (cr.pol != POL_DF) continue;
    // double-float: conditional phases on one slot that follow one another are one op, which
    // multiplies their values into one factor per thread first.  Phases commute: a run of
    // them is ordered by slot.
    for (int i = st.op0; i < st.op0 + st.nops;) {
      auto single = [&](int k) { return ops[k].type == OP_PHASE && ops[k].s0 >= 0 && !ops[k].neg; };
      if (!single(i)) {
        i++;
        continue;
      }
      int e = i;
      while (e < st.op0 + st.nops && single(e)) e++;
      std::stable_sort(ops.begin() + i, ops.begin() + e, [](const RegOp& a, const RegOp& b) { return a.s0 < b.s0; });
      for (int k = i; k < e;) {
        int m = k + 1;
        while (m < e && ops[m].s0 == ops[k].s0 && m - k < 64) m++;
        if (m - k >= 2)
          for (int q = k; q < m; q++) ops[q].s1 = (int8_t)(m - q);   // phases of the group from here on
        k = m;
      }
      i = e;
    }
  }
  return ops;
}

}  // namespace qs
