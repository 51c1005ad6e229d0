// Host emulation of the programs the tile kernels run (lowering.cpp), for the CPU tests.
//
// It compiles a circuit with the library's own compiler, lowers its register ops (lower_regops) and
// builds every pass's kernel-parameter program (build_tile_program) for a given SM count.  The passes are then
// executed in std::complex<double> with the kernels' op semantics twice: from the lowered ops with the
// plan's pool, and from the programs' bytes (stages, ops and, in double-float, the entries as lane
// patterns) where a pass has one.  Structure the kernels rely on is checked on the way and ends the
// program with an error.
//
// Usage: plan_lowering_host in.bin out.bin SMS; input as plan_emulator_host's, output int32 n, int32
// sigma_final[n], then the two states in storage order.
#define main plan_emulator_main
#include "plan_emulator_host.cpp"
#undef main

static void need(bool ok, const char* what) {
  if (ok) return;
  fprintf(stderr, "lowered program: %s\n", what);
  exit(5);
}

// One pass's program: stages and ops, and what an op's entry index stands for.
struct Program {
  const StageRec* stages;
  const RegOp* ops;
  const double* pool;     // (re, im) pairs, or
  const float* patterns;  // double-float lane patterns, 8 floats per entry
  int nops, nentries;
  C entry(int k) const {
    need(k >= 0 && k < nentries, "entry index out of range");
    if (pool) return C(pool[2 * (size_t)k], pool[2 * (size_t)k + 1]);
    const float* e = patterns + 8 * (size_t)k;
    need(e[0] == e[1] && e[2] == -e[3] && e[4] == e[5] && e[6] == -e[7], "lane patterns of an entry");
    return C((double)e[0] - (double)e[4], (double)e[3] + (double)e[7]);
  }
};

static void run_stage(std::vector<C>& x, const Program& p, const StageRec& st, int K, uint32_t gidx, uint64_t base,
                      Policy pol) {
  const bool frame = pol == POL_DF;
  const int D = 1 << K;
  for (int k = 0; k < st.nops; k++) {
    need(st.op0 + k >= 0 && st.op0 + k < p.nops, "op index out of range");
    const RegOp& op = p.ops[st.op0 + k];
    const uint32_t csl = op.csl;
    if (op.type == OP_RXTM || op.type == OP_DTAB || op.type == OP_DTAB2)
      need(op.cot == 0 && op.gmask == 0, "a table or rotation run with controls outside the registers");
    if (op.type == OP_RXTM) {
      need(csl < (uint32_t)(1 << K), "slots of a rotation run");
      int i = 0;
      for (int s = 0; s < K; s++)
        if ((csl >> s) & 1u) reg_rxt(x, s, p.entry(op.mat + i++).real(), ((uint8_t)op.neg >> s) & 1, frame);
      continue;
    }
    if (op.type == OP_DTAB) {
      for (int j = 0; j < D; j++) {
        if ((csl >> j) & 1u) x[j] *= p.entry(op.mat + j);
        else need(p.entry(op.mat + j) == C(1, 0), "a table entry outside the mask");
      }
      continue;
    }
    if (op.type == OP_DTAB2) {
      need(0 <= op.s0 && op.s0 < op.s1 && op.s1 < K, "slots of a two-slot table");
      for (int j = 0; j < D; j++)
        if (const int e = j & ((1 << op.s0) | (1 << op.s1))) x[j] *= p.entry(op.mat + e);
      continue;
    }
    if (op.type == OP_PHASE && op.s1 > 0) {
      // a group: its members count down to the last one, which has 1
      need(frame, "a group of phases outside double-float plans");
      need(k + op.s1 <= st.nops, "a group of phases past its stage");
      const int last = k + op.s1 - 1;
      for (; k <= last; k++) {
        const RegOp& o = p.ops[st.op0 + k];
        need(o.type == OP_PHASE && o.s0 == op.s0 && !o.neg && o.s1 == last - k + 1 && o.csl == 1u << o.s0,
             "a member of a group of phases");
        if ((base & o.gmask) != o.gmask || (gidx & o.cot) != o.cot) continue;
        for (int j = 0; j < D; j++)
          if ((j >> o.s0) & 1) x[j] *= p.entry(o.mat);
      }
      k = last;
      continue;
    }
    if ((base & op.gmask) != op.gmask || (gidx & op.cot) != op.cot) continue;
    if (op.type == OP_PHASE) {
      if (op.s0 >= 0) need(op.s0 < K && csl == 1u << op.s0, "slot of a phase");
      for (int j = 0; j < D; j++) {
        if (((uint32_t)j & csl) != csl) continue;
        x[j] = op.neg ? -x[j] : x[j] * p.entry(op.mat);
      }
      continue;
    }
    if (op.type == OP_RX && !p.pool) {   // from a program: entries c and s, re-based
      const double c = p.entry(op.mat).real(), sn = p.entry(op.mat + 1).real();
      for (int j = 0; j < D; j++) {
        if ((j >> op.s0) & 1) continue;
        const C a = x[j], b = x[j | (1 << op.s0)];
        x[j] = c * a + sn * b;
        x[j | (1 << op.s0)] = c * b - sn * a;
      }
      continue;
    }
    need(p.pool != nullptr || op.type == OP_X, "an op kind a program has no form of");
    Pool whole;   // the other kinds are as the compiler made them
    if (p.pool) whole.f64.assign(p.pool, p.pool + 2 * (size_t)p.nentries);
    reg_op(x, op, whole, gidx, base, frame);
  }
}

static void run_program(std::vector<C>& psi, const CompileResult& cr, const TilePass& tp, const Program& p) {
  const int L = tp.L, n = tp.n;
  const bool frame = cr.pol == POL_DF;
  const uint64_t nt = 1ull << L;
  std::vector<C> T(nt), out(psi.size());
  std::vector<uint64_t> addr(nt);
  for (uint64_t b = 0; b < 1ull << (n - L); b++) {
    uint64_t base = 0;
    for (int k = 0; k < n - L; k++)
      if (bit(b, k)) base |= 1ull << tp.npos[k];
    for (uint64_t i = 0; i < nt; i++) {
      addr[i] = base;
      for (int k = 0; k < L; k++)
        if (bit(i, k)) addr[i] |= 1ull << tp.tpos[k];
      T[i] = psi[addr[i]] * (frame ? mi_pow(popc(i)) : C(1, 0));
    }
    for (int s = tp.st0; s < tp.st0 + tp.nst; s++) {
      const StageRec& st = p.stages[s];
      if (st.kind == 1) {
        for (int o = st.op0; o < st.op0 + st.nops; o++) dev_op(T, cr.tile_ops[o], cr.pool, base, true, frame);
        continue;
      }
      const int K = popc((uint32_t)st.rmask);
      need(K == tp.K, "register bits of a stage");
      std::vector<C> x(1u << K);
      for (uint64_t g = 0; g < nt; g++) {
        if (g & (uint32_t)st.rmask) continue;
        auto at = [&](int j) {
          uint64_t i = g;
          for (int t = 0; t < K; t++)
            if ((j >> t) & 1) i |= 1ull << st.rbits[t];
          return i;
        };
        for (int j = 0; j < (1 << K); j++) x[j] = T[at(j)];
        run_stage(x, p, st, K, (uint32_t)g, base, cr.pol);
        for (int j = 0; j < (1 << K); j++) T[at(j)] = x[j];
      }
    }
    for (uint64_t i = 0; i < nt; i++) {
      const uint64_t d = ((addr[i] >> tp.swap_a) ^ (addr[i] >> tp.swap_b)) & 1ull;
      out[addr[i] ^ ((d << tp.swap_a) | (d << tp.swap_b))] = T[i] * (frame ? mi_pow(-popc(i)) : C(1, 0));
    }
  }
  psi.swap(out);
}

// the view of a program's bytes; its ops must fill the space between the stages and the entries
template <int NB>
static Program program_view(const CompileResult& cr, const std::vector<unsigned char>& bytes, const TilePass& tp) {
  need(bytes.size() == sizeof(TileProg<NB>), "size of a program");
  const TileProg<NB>& t = *(const TileProg<NB>*)bytes.data();
  need(t.tp.st0 == 0 && t.tp.nst == tp.nst && t.tp.L == tp.L && t.tp.n == tp.n && t.tp.K == tp.K &&
       t.tp.flags == tp.flags && t.tp.swap_a == tp.swap_a && t.tp.swap_b == tp.swap_b &&
       !memcmp(t.tp.tpos, tp.tpos, sizeof tp.tpos) && !memcmp(t.tp.npos, tp.npos, sizeof tp.npos), "a program's pass");
  need(t.off_ops >= (int)(tp.nst * sizeof(StageRec)) && t.off_ops % 16 == 0 && t.off_pool % 16 == 0 &&
       t.off_pool <= NB, "a program's offsets");
  Program p{};
  p.stages = (const StageRec*)t.data;
  p.ops = (const RegOp*)(t.data + t.off_ops);
  p.nops = (t.off_pool - t.off_ops) / (int)sizeof(RegOp);
  if (cr.pol == POL_DF) {
    p.patterns = (const float*)(t.data + t.off_pool);
    p.nentries = (NB - t.off_pool) / 32;
  } else {
    p.pool = cr.pool.f64.data();
    p.nentries = (int)cr.pool.entries();
  }
  return p;
}

int main(int argc, char** argv) {
  if (argc != 4) return 2;
  FILE* f = fopen(argv[1], "rb");
  if (!f) return 2;
  int32_t n = 0, nops = 0, has_cost = 0;
  int64_t nmats = 0;
  qs_compile_opts o;
  qs_cost_model cost{};
  bool ok = fread(&n, 4, 1, f) == 1 && fread(&nops, 4, 1, f) == 1 && fread(&nmats, 8, 1, f) == 1 &&
            fread(&o, sizeof(o), 1, f) == 1 && fread(&has_cost, 4, 1, f) == 1 && fread(&cost, sizeof(cost), 1, f) == 1;
  o.cost = nullptr;
  std::vector<qs_op> ops(nops);
  std::vector<double> mats(nmats > 0 ? nmats : 1);
  ok = ok && (nops == 0 || fread(ops.data(), sizeof(qs_op), nops, f) == (size_t)nops);
  ok = ok && (nmats == 0 || fread(mats.data(), 8, nmats, f) == (size_t)nmats);
  fclose(f);
  std::string err;
  if (!ok || !normalize_compile_opts(n, &o, &err)) return 2;
  std::vector<HGate> gates(nops);
  for (int i = 0; i < nops; i++)
    if (!make_hgate(n, ops[i], mats.data(), (size_t)nmats, &gates[i], &err)) return 4;
  std::vector<int> sigma0(n);
  for (int q = 0; q < n; q++) sigma0[q] = q;
  CompileResult cr;
  if (!compile_circuit(n, gates, sigma0, o, &cr, &err)) return 4;

  const int sms = atoi(argv[3]);
  const std::vector<RegOp> rops = lower_regops(cr);
  need(rops.size() == cr.reg_ops.size(), "number of ops");
  Program arrays{};
  arrays.stages = cr.stages.data();
  arrays.ops = rops.data();
  arrays.nops = (int)rops.size();
  arrays.pool = cr.pool.f64.data();
  arrays.nentries = (int)cr.pool.entries();
  std::vector<C> a(1ull << n, C(0, 0)), b;
  a[0] = 1;
  b = a;
  int passes = 0, programs = 0;
  for (const Step& s : cr.steps) {
    if (s.kind != ST_PASS) return 6;   // the tests' plans hold passes only
    passes++;
    run_program(a, cr, s.pass, arrays);
    std::vector<unsigned char> prog;
    if (!build_tile_program(cr, rops, s.pass, sms, &prog)) {
      need(prog.empty(), "bytes of a refused program");
      run_program(b, cr, s.pass, arrays);
      continue;
    }
    programs++;
    TilePass tp = s.pass;
    const Program p = cr.pol == POL_DF ? program_view<kTileProgDF>(cr, prog, tp) : program_view<kTileProgF32>(cr, prog, tp);
    tp.st0 = 0;
    run_program(b, cr, tp, p);
  }
  int dtab2 = 0, slot = 0, grouped = 0;   // ops of the lowered kinds
  for (const RegOp& r : rops) {
    dtab2 += r.type == OP_DTAB2;
    slot += r.type == OP_PHASE && r.s0 >= 0 && r.s1 <= 0;
    grouped += r.type == OP_PHASE && r.s1 > 0;
  }
  fprintf(stderr, "passes %d programs %d dtab2 %d slot %d grouped %d\n", passes, programs, dtab2, slot, grouped);
  FILE* g = fopen(argv[2], "wb");
  if (!g) return 2;
  fwrite(&n, 4, 1, g);
  for (int q = 0; q < n; q++) {
    const int32_t v = cr.sigma_final.empty() ? q : cr.sigma_final[q];
    fwrite(&v, 4, 1, g);
  }
  fwrite(a.data(), sizeof(C), a.size(), g);
  fwrite(b.data(), sizeof(C), b.size(), g);
  fclose(g);
  return 0;
}
