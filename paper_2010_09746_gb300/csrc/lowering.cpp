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
#include <string.h>

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

namespace {

// consecutive matrix entries a double-float op reads from its mat on
int entries_of(const RegOp& r, int K) {
  switch (r.type) {
    case OP_DTAB: return 1 << K;
    case OP_DTAB2: return ((1 << r.s0) | (1 << r.s1)) + 1;
    case OP_RXTM: return __builtin_popcount(r.csl);
    case OP_RX: return 2;   // c and s apart
    case OP_PHASE: return r.neg ? 0 : 1;
    default: return 0;
  }
}

template <int NB>
bool build_program(const CompileResult& cr, const std::vector<RegOp>& ops, const TilePass& tp,
                   std::vector<unsigned char>* out) {
  const bool entries = cr.pol == POL_DF;
  size_t nops = 0, nent = 0;
  for (int k = tp.st0; k < tp.st0 + tp.nst; k++) {
    const StageRec& st = cr.stages[k];
    if (st.kind != 0) return false;
    nops += st.nops;
    for (int i = st.op0; i < st.op0 + st.nops; i++) {
      const RegOp& r = ops[i];
      const bool known = r.type == OP_RXTM || r.type == OP_DTAB || r.type == OP_DTAB2 || r.type == OP_PHASE ||
                         r.type == OP_RX || r.type == OP_X;
      if (!known) return false;
      nent += entries ? entries_of(r, tp.K) : 0;
    }
  }
  const size_t off_ops = (tp.nst * sizeof(StageRec) + 15) & ~(size_t)15, off_pool = off_ops + nops * sizeof(RegOp);
  const size_t eb = Pool::entry_bytes(cr.pol);
  if (off_pool + nent * eb > (size_t)NB) return false;
  out->assign(sizeof(TileProg<NB>), 0);
  TileProg<NB>& p = *(TileProg<NB>*)out->data();
  p.tp = tp;
  p.tp.st0 = 0;
  p.off_ops = (int32_t)off_ops;
  p.off_pool = (int32_t)off_pool;
  StageRec* sts = (StageRec*)p.data;
  RegOp* dst = (RegOp*)(p.data + off_ops);
  float* pool = (float*)(p.data + off_pool);
  int o = 0, e = 0;
  for (int k = 0; k < tp.nst; k++) {
    sts[k] = cr.stages[tp.st0 + k];
    const int op0 = sts[k].op0;
    sts[k].op0 = o;
    for (int i = op0; i < op0 + sts[k].nops; i++) {
      RegOp r = ops[i];
      if (entries) {
        const int ne = entries_of(r, tp.K);
        for (int q = 0; q < ne; q++) df_entry(&cr.pool.f64[2 * ((size_t)r.mat + q)], pool + 8 * (e + q));
        r.mat = e;
        e += ne;
      }
      dst[o++] = r;
    }
  }
  return true;
}

}  // namespace

// A program in the kernel parameters is used for complex64, but for passes without moves over many tiles,
// and for double-float with no more tiles than SMs (one CTA on an SM).  Constant-bank ops decode in uniform
// registers, and the kernel holds none of the rarer ops' code.  Measured, device arrays against parameters:
// complex64 Haar circuits of 14 / 17 / 20 / 23 qubits 961 / 1142 / 1518 / 6111 -> 765 / 923 / 1218 / 5298 us, Algorithm 1
// at 26 qubits 48.6 -> 45.9 ms.  Passes without moves have a light device-array kernel; RZ / RX / CZ circuits of
// 13 / 18 / 22 / 24 / 26 qubits 169 / 310 / 851 / 3247 / 12216 -> 143 / 267 / 782 / 3157 / 12208 us, but 27 and 28 qubits (2^14 and
// 2^15 tiles) 24.77 / 31.01 -> 24.89 / 31.25 ms and QFTs of 27 / 29 qubits 11.66 / 50.15 -> 11.84 / 52.12 ms (Algorithm 1 at
// 27 qubits, whose passes are short, 77.28 -> 77.06): with 50 tiles and more per CTA the program's start no longer counts.
// Double-float at 16 / 18 qubits (16 / 64 tiles) 1417 / 1623 -> 1280 / 1457 us
// (1096 / 1242 since the kernel has an SM's registers for one CTA), but at 20 qubits (256 tiles) 2076 -> 2246 us
// and at 23 qubits 15.9 -> 17.0 ms: two CTAs on an SM run through 9 to 30 KB of entries each, past the
// constant cache.  With ops alone in parameters double-float lost 4 %
// everywhere, and complex64 entries there lost 8 % at 27 qubits.
bool build_tile_program(const CompileResult& cr, const std::vector<RegOp>& ops, const TilePass& tp, int sms,
                        std::vector<unsigned char>* out) {
  out->clear();
  if (tp.nst == 0) return false;
  const bool light_and_many = (tp.flags & kPassLite) && tp.n - tp.L >= 14;
  if (cr.pol == POL_F32 && tp.K == 5 && !light_and_many) return build_program<kTileProgF32>(cr, ops, tp, out);
  if (cr.pol == POL_DF && tp.K == 4 && tp.n - tp.L < 31 && (1 << (tp.n - tp.L)) <= sms)
    return build_program<kTileProgDF>(cr, ops, tp, out);
  return false;
}

}  // namespace qs
