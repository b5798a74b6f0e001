// pc_jit.cpp -- run-time specialised pricing kernels.
//
// The paper compiles each contract to a payoff function of its own (Sec. 6:
// Futhark code per instrument).  The engine's default kernel interprets the
// executable program instead, which costs a dispatch per instruction.  Here
// the program is turned into straight-line CUDA: one labelled block per
// instruction, each the interpreter's case for that opcode (the text of
// pc_ops.inc, split per opcode at build time), with NEXT / JUMP_* as gotos
// between the blocks.  The block bodies are the
// interpreter's own text, so both evaluators compute the same operations in
// the same order.  NVRTC compiles the module for the device the context
// runs on; the kernel is price_tiles (pc_price.cuh) with this evaluator.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <sstream>
#include <string>
#include <thread>
#include <vector>

#include <nvrtc.h>

#include "pc_handles.h"
#include "pc_internal.h"
#include "pc_cv_types.h"
#include "pc_jit_headers.inc"

using namespace pc;

namespace {

std::string hex(uint32_t v) {
  char b[16];
  std::snprintf(b, sizeof(b), "0x%08xu", v);
  return b;
}

// The interpreter's case for an opcode (pc_ops.inc, split by the build);
// unknown opcodes take the default case (return), as in the interpreter.
const char *case_text(uint32_t op) {
  return op < uint32_t(kJitCaseCount) ? kJitCase[op] : kJitCase[0];
}

std::string insn_literal(const XInsn &I) {
  return "make_uint4(" + hex(I.opa) + ", " + hex(I.b) + ", " + hex(I.c) + ", " + hex(I.e) + ")";
}

// Above this many reading instructions a program whose stack depths are
// not known calls the date generator out of line.
constexpr int kInlineDateSites = 12;
// Above this many reading instructions the re-entry switch of the shared
// generator makes NVRTC's time grow faster than the program (100 terms of
// a two-asset average: 13 s shared, 3.2 s out of line): call it out of line.
constexpr int kSharedDateSites = 64;
// The adjoint evaluator's code grows by its tape writes at every operation:
// an average of 3 / 6 / 12 / 27 / 50 reads compiles in 1.3 / 1.8 / 2.2 / 6.4 /
// 24.6 s (its pricing kernel in 0.4 to 1.1).  Longer ones are interpreted; the
// limit dates from a generator inlined at each read, and where it would lie
// best with the shared one has not been measured.
constexpr int kAdjointDateSites = 6;
// Instructions that read simulated dates (and may have to generate them).
bool reads_dates(const XInsn &I) {
  const uint32_t op = I.opa & 0xffu;
  return op == X_MODEL || op == X_MODEL_MULK || op == X_MODEL_DIVK || op == X_LRED || op == X_LANY;
}

int date_sites(const Program &p) {
  int n = 0;
  for (const XInsn &I : p.code) n += reads_dates(I);
  return n;
}

// The evaluator's operand-stack pointer (sp) before each instruction, from
// every opcode's effect on each of its exits (the cases of pc_ops.inc):
// -1 for instructions no path reaches.  False when an opcode has no known
// effect, a depth leaves [0, frame_slots), or two paths meet with different
// depths -- the program is then specialised without re-entry points.
bool stack_depths(const Program &p, std::vector<int> &sp_at) {
  const int n = int(p.code.size());
  sp_at.assign(size_t(n), -1);
  if (n == 0) return false;
  std::vector<int> work;
  bool ok = true;
  auto flow = [&](uint32_t t, int v) {
    if (t >= uint32_t(n) || v < 0 || v >= std::max(1, int(p.frame_slots))) {
      ok = false;
      return;
    }
    if (sp_at[t] < 0) {
      sp_at[t] = v;
      work.push_back(int(t));
    } else if (sp_at[t] != v) {
      ok = false;
    }
  };
  flow(0, 0);
  while (ok && !work.empty()) {
    const int i = work.back();
    work.pop_back();
    const XInsn &I = p.code[size_t(i)];
    const int s = sp_at[size_t(i)];
    const uint32_t nx = uint32_t(i + 1);
    switch (I.opa & 0xffu) {
      case X_END: break;
      case X_CONST: case X_MODEL: case X_PAYOFF: case X_TIME: case X_NOW: case X_MODEL_MULK:
      case X_MODEL_DIVK: case X_LRED: case X_LANY:
        flow(nx, s + 1);
        break;
      case X_NEGF: case X_NOT: case X_ADDFK: case X_SUBFK: case X_MULFK: case X_DIVFK: case X_MAXFK:
      case X_MINFK: case X_LTFK: case X_LEFK: case X_EQFK: case X_RSUBFK: case X_RDIVFK: case X_RLTFK:
      case X_RLEFK: case X_LOOP: case X_LEND:
        flow(nx, s);
        break;
      case X_ADDF: case X_SUBF: case X_MULF: case X_DIVF: case X_MAXF: case X_MINF: case X_LTF: case X_LEF:
      case X_EQF: case X_ADDI: case X_SUBI: case X_MULI: case X_MAXI: case X_MINI: case X_LTI: case X_LEI:
      case X_EQI: case X_AND: case X_OR: case X_LLATCH:
        flow(nx, s - 1);
        break;
      case X_SEL: flow(nx, s - 2); break;
      case X_IF: case X_ELSE:  // NEXT, or push a placeholder and JUMP_Z
        flow(nx, s);
        flow(I.c, s + 1);
        break;
      case X_LTEST:  // pop; NEXT or JUMP_Z
        flow(nx, s - 1);
        flow(I.c, s - 1);
        break;
      case X_LSTEPK:  // pop; push the result and JUMP_W, NEXT, or JUMP_Z
        flow(I.e, s);
        flow(nx, s - 1);
        flow(I.c, s - 1);
        break;
      case X_LNEXT:
        flow(I.e, s + 1);
        flow(nx, s);
        flow(I.c, s);
        break;
      case X_LOOPANY:  // push the result and JUMP_W, or JUMP_2 (pc + 1 is a descriptor)
        flow(I.e, s + 1);
        flow(uint32_t(i + 2), s);
        break;
      default: ok = false; break;
    }
  }
  return ok;
}

// A price or control-variate evaluator without re-entry points: many reading
// instructions call one out-of-line copy of the generator instead of
// inlining it at each.
bool outlined_dates(const Program &p) {
  std::vector<int> sp_at;
  const bool shared = date_sites(p) >= 2 && date_sites(p) <= kSharedDateSites && stack_depths(p, sp_at);
  return !shared && date_sites(p) > kInlineDateSites;
}

// A static walk as source: PC_STEP runs step ps.step (its ops, then its date).
// Defined before the device headers, whose state it sizes.
void define_walk(std::ostringstream &o, const JitSpec &sp) {
  auto ints = [&](const char *name, const std::vector<int32_t> &v) {
    if (v.empty()) return;
    o << "#define " << name;
    for (size_t i = 0; i < v.size(); ++i) o << (i ? ", " : " ") << v[i];
    o << "\n";
  };
  ints("PC_LAYOUT", sp.lay);
  ints("PC_GRID", sp.grid);
  if (sp.walk.empty()) return;
  int depth = 1, bsp = 0, idx = 0, cur = -1;
  size_t steps = 0;
  for (size_t i = 0; i < sp.walk.size(); ++steps) {
    const int date = sp.walk[i], read = sp.walk[i + 1], ops = sp.walk[i + 2];
    i += 3;
    o << "#define PC_STEP_" << steps << "(XW_, GW_, LM_) { \\\n";
    for (int j = 0; j < ops; ++j, ++i, ++idx, ++bsp) {
      const int k = sp.walk[i];
      o << "      static_op<D, PC_PAIRS, " << k << ", " << idx << ", " << bsp << ", " << cur << ">(ps, g, sg); \\\n";
      cur = (sp.d * k + sp.d - 1) / 4;
    }
    depth = std::max(depth, bsp);
    --bsp;
    o << "      static_date<D, PC_PAIRS, XW_, GW_, " << steps << ", " << bsp << ", " << (read ? "true" : "false")
      << ">(" << date << ", ps, lay, sg, R, Bm, S0, LM_); }\n";
  }
  o << "#define PC_STATIC_DEPTH " << depth << "\n"
    << "#define PC_STEP(XW_, GW_, LM_) switch (ps.step) { \\\n";
  for (size_t i = 0; i < steps; ++i) o << "    case " << i << ": PC_STEP_" << i << "(XW_, GW_, LM_) break; \\\n";
  o << "    default: ps.f = 0x7fffffff; }\n";
}

// With a static walk: what every run has at an instruction, by data flow over
// the program -- the loop offset t0 and the frontier (the last date produced),
// each known or not (kUnknown) where paths of different history meet or a
// loop is under way.  A reading instruction with both known runs exactly the
// steps from its frontier to its date in line: no test, no jump, one copy in
// programs that read each date first at one place.
constexpr int kUnknown = -(1 << 30);
struct FlowState {
  int t0 = 0, f = 0;
  bool reached = false;
};
std::vector<FlowState> flow_states(const Program &p, const JitSpec &sp) {
  const int n = int(p.code.size()), t_now = sp.grid[2];
  std::vector<FlowState> at(static_cast<size_t>(n));
  std::vector<int> lend_t0(static_cast<size_t>(n), kUnknown), work;
  auto flow = [&](uint32_t t, int t0, int f) {
    if (t >= uint32_t(n)) return;
    FlowState &x = at[t];
    const int nt0 = !x.reached || x.t0 == t0 ? t0 : kUnknown, nf = !x.reached || x.f == f ? f : kUnknown;
    if (x.reached && nt0 == x.t0 && nf == x.f) return;
    x = {nt0, nf, true};
    work.push_back(int(t));
  };
  flow(0, 0, 0);
  while (!work.empty()) {
    const int i = work.back();
    work.pop_back();
    const XInsn &I = p.code[size_t(i)];
    const int t0 = at[size_t(i)].t0;
    int f = at[size_t(i)].f;
    const uint32_t nx = uint32_t(i + 1), op = I.opa & 0xffu;
    if (reads_dates(I)) {
      if (t0 == kUnknown) f = kUnknown;
      else if (f != kUnknown) f = std::max(f, int(I.b) + t0 - t_now);
      flow(nx, t0, f);
      continue;
    }
    switch (op) {
      case X_END: break;
      case X_IF: case X_ELSE:
        flow(nx, t0, f);
        flow(I.c, t0, f);
        break;
      case X_LOOPANY: {
        const int last = t0 == kUnknown ? kUnknown : int(p.code[size_t(i) + 1].b) + t0 + int(I.b) - t_now;
        lend_t0[I.e - 1] = t0;
        flow(I.e, t0, kUnknown);  // every path latched, at any of its dates
        flow(uint32_t(i + 2), t0 == kUnknown ? kUnknown : t0 + int(I.b),
             f == kUnknown || last == kUnknown ? kUnknown : std::max(f, last));
        break;
      }
      case X_LEND: flow(nx, lend_t0[size_t(i)], f); break;
      case X_LOOP: case X_LTEST: case X_LLATCH: case X_LNEXT: case X_LSTEPK:
        flow(nx, kUnknown, kUnknown);
        flow(I.c, kUnknown, kUnknown);
        flow(I.e, kUnknown, kUnknown);
        break;
      default: flow(nx, t0, f); break;
    }
  }
  return at;
}
// The ENSURE of a reading instruction whose state is known (false if it is
// not): the steps to its date.
bool known_ensure(const XInsn &I, const FlowState &st, const JitSpec &sp, const char *args, std::string &text) {
  if (!st.reached || st.t0 == kUnknown || st.f == kUnknown) return false;
  const int target = int(I.b) + st.t0 - sp.grid[2];
  text = "#define ENSURE(o) {";
  int step = 0;
  for (size_t i = 0; i < sp.walk.size(); i += 3 + size_t(sp.walk[i + 2]), ++step)
    if (sp.walk[i] > st.f && sp.walk[i] <= target) {
      text += " PC_STEP_" + std::to_string(step) + args;
      if (sp.kind >= kJitCv && sp.kind < kJitGreeks) text += " hook_->on_date(" + std::to_string(sp.walk[i]) + ", read);";
    }
  text += " }\n";
  return true;
}

// A static walk's launch argument, as a kernel and as an evaluator parameter.
const char *walk_kernel_param(const JitSpec &sp) { return sp.walk.empty() ? "" : ", const __grid_constant__ pc::StaticGrid sg"; }
const char *walk_eval_param(const JitSpec &sp) { return sp.walk.empty() ? "" : ", const StaticGrid &sg"; }
const char *walk_arg(const JitSpec &sp) { return sp.walk.empty() ? "" : ", sg"; }

// The program's constant pool as literals.
void define_pool(std::ostringstream &o, const Program &p) {
  o << "__device__ constexpr float kPool[] = {0.f";
  char b[40];
  for (float f : p.pool) {
    if (f - f == 0.f) std::snprintf(b, sizeof(b), ", %af", double(f));
    else std::snprintf(b, sizeof(b), ", %s", f != f ? "__builtin_nanf(\"\")" : f > 0 ? "__builtin_huge_valf()" : "-__builtin_huge_valf()");
    o << b;
  }
  o << "};\n#define pool (kPool + 1)\n";
}

// One copy of the date generator for the program's reading instructions: a
// reading instruction that needs dates jumps to PC_GEN and it jumps back to
// the top of that instruction (`resume` restores its static state).
template <typename RESUME>
void shared_generator(std::ostringstream &o, const Program &p, const std::vector<std::string> &known,
                      const char *advance, RESUME resume) {
  bool any = false;
  for (size_t i = 0; i < p.code.size(); ++i) any = any || (reads_dates(p.code[i]) && known[i].empty());
  if (!any) return;
  o << "  int need_ = 0, resume_ = -1;\n"
    << "  goto L0;\n"
    << "PC_GEN:\n"
    << "  " << advance << "\n"
    << "  switch (resume_) {\n";
  for (size_t i = 0; i < p.code.size(); ++i)
    if (reads_dates(p.code[i]) && known[i].empty()) resume(i);
  o << "    default: return tos;\n"
    << "  }\n";
}
// Per instruction the ENSURE text of a reading instruction whose state is
// known; empty for the others (and without a walk).
std::vector<std::string> known_sites(const Program &p, const JitSpec &sp, const char *args) {
  std::vector<std::string> known(p.code.size());
  if (sp.walk.empty()) return known;
  const std::vector<FlowState> at = flow_states(p, sp);
  for (size_t i = 0; i < p.code.size(); ++i)
    if (reads_dates(p.code[i])) known_ensure(p.code[i], at[i], sp, args, known[i]);
  return known;
}
std::string shared_ensure(size_t i) {
  return "#define ENSURE(o) { if ((o) > m.n || (o) < -m.n_hist) { atomicOr(a.status, 1); "
         "(o) = (o) > m.n ? m.n : -m.n_hist; } if (ps.f < (o)) { need_ = (o); resume_ = " +
         std::to_string(i) + "; goto PC_GEN; } }\n";
}

// The sensitivity evaluators straight-line over the program: each
// instruction is the interpreter's case for its constant opcode and fields
// (ops_inc), followed by a jump to whichever of its possible successors the
// case left in pc.  The operand stack stays in shared memory, as in the
// interpreter, so the shared date generator needs no stack depths.
void sensitivity_blocks(std::ostringstream &o, const Program &p, const JitSpec &sp, const char *ops_inc,
                        const char *end) {
  const size_t n = p.code.size();
  const bool shared = date_sites(p) >= 2;
  const std::vector<std::string> known = known_sites(p, sp, "(true, false, Lm)");
  if (shared)
    shared_generator(o, p, known, "while (ps.f < need_) NEXT_DATE(true, false, Lm);",
                     [&](size_t i) { o << "    case " << i << ": goto L" << i << ";\n"; });
  o << "  goto L0;\n";
  for (size_t i = 0; i < n; ++i) {
    const XInsn &I = p.code[i];
    o << "L" << i << ": {\n"
      << "  pc = " << i << ";\n"
      << "  const uint4 I = " << insn_literal(I) << ";\n"
      << "  const uint32_t op = " << hex(I.opa & 0xffu) << ";\n"
      << "  const float kk = __uint_as_float(" << hex(I.b) << ");\n"
      << "#define NEXT_INSN " << insn_literal(i + 1 < n ? p.code[i + 1] : I) << "\n"
      << (!known[i].empty() ? known[i]
          : shared && reads_dates(I) ? shared_ensure(i) : std::string("#define ENSURE(o) ensure(o)\n"))
      << "#include \"" << ops_inc << "\"\n"
      << "#undef ENSURE\n#undef NEXT_INSN\n";
    std::vector<uint32_t> next = {uint32_t(i + 1), I.c, I.e, uint32_t(i + 2)};
    for (size_t j = 0; j < next.size(); ++j) {
      bool seen = false;
      for (size_t q = 0; q < j; ++q) seen = seen || next[q] == next[j];
      if (!seen && next[j] < n) o << "  if (pc == " << next[j] << ") goto L" << next[j] << ";\n";
    }
    o << end << "  return tos;\n"
      << "}\n";
  }
}

// pc_jit_adjoint: adjoint_tiles around the specialised adjoint evaluator.
std::string generate_adjoint(const Program &p, const JitSpec &sp, bool write) {
  std::ostringstream o;
  define_walk(o, sp);
  o << "#include \"pc_adjoint.cuh\"\n"
    << "namespace pc {\n"
    << "namespace {\n"
    << "constexpr int D = " << sp.d << ";\n";
  define_pool(o, p);
  o << "__device__ __forceinline__ float2 jit_eval_adjoint(const uint4 *P, float2 *R,\n"
    << "    const PriceArgs &a, const Rng2 &g, bool live0, bool live1, const float (&Bm)[D * D],\n"
    << "    const float (&S0)[D], const float (&Lm)[D * D], Tape &T, int &res" << walk_eval_param(sp) << ") {\n"
    << "#include \"pc_adjoint_state.inc\"\n";
  sensitivity_blocks(o, p, sp, "pc_adjoint_ops.inc", "  res = tid;\n");
  o << "}\n"
    << "#undef pool\n"
    << "}  // namespace\n"
    << "}  // namespace pc\n"
    << "extern \"C\" __global__ void __launch_bounds__(" << kBlock
    << ") pc_jit_adjoint(const __grid_constant__ pc::PriceArgs a, const pc::TapeArgs t" << walk_kernel_param(sp) << ") {\n"
    << "  pc::adjoint_tiles<pc::D, " << (write ? "true" : "false") << ">(a, t, [&](const uint4 *P, const float *,\n"
    << "      float2 *R, const pc::Rng2 &g, bool live0, bool live1, const float (&Bm)[pc::D * pc::D],\n"
    << "      const float (&S0)[pc::D], const float (&Lm)[pc::D * pc::D], pc::Tape &T, int &res) {\n"
    << "    return pc::jit_eval_adjoint(P, R, a, g, live0, live1, Bm, S0, Lm, T, res" << walk_arg(sp) << "); });\n"
    << "}\n";
  return o.str();
}

// pc_jit_greeks: greeks_tiles around the specialised tangent evaluator (the
// per-path triples written out with kJitGreeks + 1).
std::string generate_greeks(const Program &p, const JitSpec &sp, bool write) {
  std::ostringstream o;
  define_walk(o, sp);
  o << "#include \"pc_greeks.cuh\"\n"
    << "namespace pc {\n"
    << "namespace {\n"
    << "constexpr int D = " << sp.d << ";\n";
  define_pool(o, p);
  o << "__device__ __forceinline__ TV jit_eval_greeks(const uint4 *P, float2 *R,\n"
    << "    const PriceArgs &a, const Rng2 &g, bool live0, bool live1, const float (&Bm)[D * D],\n"
    << "    const float (&S0)[D], const float (&Lm)[D * D], int gl, float sig_g" << walk_eval_param(sp) << ") {\n"
    << "#include \"pc_greeks_state.inc\"\n";
  sensitivity_blocks(o, p, sp, "pc_greeks_ops.inc", "");
  o << "}\n"
    << "#undef pool\n"
    << "}  // namespace\n"
    << "}  // namespace pc\n"
    << "extern \"C\" __global__ void __launch_bounds__(" << kBlock
    << ") pc_jit_greeks(const __grid_constant__ pc::PriceArgs a" << walk_kernel_param(sp) << ") {\n"
    << "  pc::greeks_tiles<pc::D, " << (write ? "true" : "false") << ">(a, [&](const uint4 *P, const float *,\n"
    << "      float2 *R, const pc::Rng2 &g, bool live0, bool live1, const float (&Bm)[pc::D * pc::D],\n"
    << "      const float (&S0)[pc::D], const float (&Lm)[pc::D * pc::D], int gl, float sig_g) {\n"
    << "    return pc::jit_eval_greeks(P, R, a, g, live0, live1, Bm, S0, Lm, gl, sig_g" << walk_arg(sp) << "); });\n"
    << "}\n";
  return o.str();
}

// Straight-line evaluator for the program and d underlyings, and the kernel
// of `kind` around it: pc_jit_price (price_tiles; per-path payoffs written
// out with kJitPriceWrite, the window of dates in HBM with kJitHbm) or
// pc_jit_cv (cv_tiles with mode kind - kJitCv).
// With two or more reading instructions and known stack depths, the date
// generator has one copy: a reading instruction that needs dates jumps to
// it and it jumps back to the top of that instruction, restoring the
// static stack pointer there (so the operand stack stays in registers).
// Otherwise the generator is inlined at each reading instruction (out of
// line beyond kInlineDateSites of them).
std::string generate(const Program &p, const JitSpec &spec) {
  const int d = spec.d, kind = spec.kind;
  if (kind >= kJitAdjoint) return generate_adjoint(p, spec, (kind & 1) != 0);
  if (kind >= kJitGreeks) return generate_greeks(p, spec, (kind & 1) != 0);
  std::ostringstream o;
  const size_t n = p.code.size();
  std::vector<int> sp_at;
  const bool shared = date_sites(p) >= 2 && date_sites(p) <= kSharedDateSites && stack_depths(p, sp_at);
  if (outlined_dates(p)) o << "#define PC_JIT_OUTLINE_DATES 1\n";
  define_walk(o, spec);
  // a program that reads no date behind the frontier keeps that date's S in
  // registers instead of a shared-memory window
  if ((kind < kJitCv && (kind & kJitWinRegs)) || (kind >= kJitCv && ((kind - kJitCv) & kCvWinRegs)))
    o << "#define PC_WIN_REGS 1\n";
  // four paths a lane: the per-op and per-instruction control serves twice
  // the paths
  const bool pairs2 = kind < kJitCv && (kind & kJitPairs2);
  if (pairs2) o << "#define PC_PAIRS 2\n";
  o << "#include \"pc_price.cuh\"\n";
  if (kind >= kJitCv) o << "#include \"pc_cv.cuh\"\n";
  o
    << "namespace pc {\n"
    << "namespace {\n"
    << "constexpr int D = " << d << ";\n"
    << "constexpr bool GW = " << (kind < kJitCv && (kind & kJitHbm) ? "true" : "false") << ";\n"
    << "#define PC_JIT_STACK_SLOTS " << std::max(1, int(p.frame_slots)) << "\n";
  define_pool(o, p);
  o << "template <class PcHook = NoDateHook>\n"
    << "__device__ __forceinline__ PV jit_eval(const uint4 *P, float2 *R,\n"
    << (pairs2 ? "    const PriceArgs &a, const RngH<2> &g, const bool (&live_)[kPL], const float (&Bm)[D * D],\n"
               : "    const PriceArgs &a, const Rng2 &g, bool live0, bool live1, const float (&Bm)[D * D],\n")
    << "    const float (&S0)[D]" << walk_eval_param(spec) << ", int *frontier = nullptr, PcHook *hook_ = nullptr) {\n"
    << "#include \"pc_eval_state.inc\"\n"
    << "  (void)pc;\n";
  const std::vector<std::string> known =
      known_sites(p, spec, kind < kJitCv && (kind & kJitHbm) ? "(false, true, nullptr)" : "(false, false, nullptr)");
  if (shared)
    shared_generator(o, p, known, "EACH_DATE(need_)", [&](size_t i) {
      if (sp_at[i] >= 0) o << "    case " << i << ": sp = " << sp_at[i] << "; goto L" << i << ";\n";
    });
  for (size_t i = 0; i < n; ++i) {
    const XInsn &I = p.code[i];
    const size_t nx = i + 1 < n ? i + 1 : i;
    auto lbl = [&](size_t t) { return "L" + std::to_string(t < n ? t : n - 1); };
    o << lbl(i) << ": {\n"
      << "#define NEXT { goto " << lbl(nx) << "; }\n"
      << "#define JUMP_Z { goto " << lbl(I.c) << "; }\n"
      << "#define JUMP_W { goto " << lbl(I.e) << "; }\n"
      << "#define JUMP_2 { goto " << lbl(i + 2) << "; }\n"
      << "#define NEXT_INSN " << (i + 1 < n ? insn_literal(p.code[i + 1]) : insn_literal(I)) << "\n";
    if (!known[i].empty())
      o << known[i];
    else if (shared && reads_dates(I) && sp_at[i] >= 0)
      o << shared_ensure(i);
    else
      o << "#define ENSURE(o) ensure(o)\n";
    o << "  const uint4 I = " << insn_literal(I) << ";\n"
      << "  {\n" << case_text(I.opa & 0xffu) << "  }\n"
      << "#undef NEXT\n#undef JUMP_Z\n#undef JUMP_W\n#undef JUMP_2\n#undef NEXT_INSN\n#undef ENSURE\n"
      << "}\n";
  }
  o << "  return tos;\n"
    << "#undef PUSH\n#undef STK\n#undef BINF\n#undef BINI\n#undef IMM\n#undef EACH_DATE\n#undef pool\n"
    << "}\n"
    << "}  // namespace\n"
    << "}  // namespace pc\n";
  if (kind >= kJitCv) {
    // the register bound (PC_MIN_BLOCKS resident blocks) is passed by the
    // launcher
    const bool gamma = ((kind - kJitCv) & kCvGamma) != 0;
    o << "#ifndef PC_MIN_BLOCKS\n#define PC_MIN_BLOCKS " << kJitCvMinBlocks << "\n#endif\n"
      << "extern \"C\" __global__ void __launch_bounds__(" << kBlock
      << ", PC_MIN_BLOCKS) pc_jit_cv(const __grid_constant__ pc::PriceArgs a,\n"
      << "    const __grid_constant__ pc::CvArgs c" << walk_kernel_param(spec) << ") {\n"
      << "  using Hook = pc::CvOnline<pc::D, " << (gamma ? "true" : "false") << ">;\n"
      << "  pc::cv_tiles<pc::D, " << ((kind - kJitCv) & 7) << ">(a, c, [&](const uint4 *P, const float *, float2 *R,\n"
      << "      const pc::Rng2 &g, bool live0, bool live1, const float (&Bm)[pc::D * pc::D],\n"
      << "      const float (&S0)[pc::D], Hook *hook) {\n"
      << "    return pc::jit_eval<Hook>(P, R, a, g, live0, live1, Bm, S0" << walk_arg(spec) << ", nullptr, hook); });\n"
      << "}\n";
    return o.str();
  }
  // resident 128-thread blocks per SM the register bound is set for
  // (PC_MIN_BLOCKS, passed by the launcher: 7, <= 72 registers, unless the
  // launch's shared memory already allows fewer, whose bound then leaves the
  // kernel the registers those blocks can have)
  o << "#ifndef PC_MIN_BLOCKS\n#define PC_MIN_BLOCKS " << kJitMinBlocks << "\n#endif\n"
    << "extern \"C\" __global__ void __launch_bounds__(" << kBlock << ", PC_MIN_BLOCKS) pc_jit_price(const __grid_constant__ pc::PriceArgs a" << walk_kernel_param(spec) << ") {\n";
  if (pairs2)
    o << "  pc::price_tiles2<pc::D, " << (kind & kJitPriceWrite ? "true" : "false") << ">(a, [&](const uint4 *P, const float *,\n"
      << "      float2 *R, const pc::RngH<2> &g, const bool (&live)[4], const float (&Bm)[pc::D * pc::D],\n"
      << "      const float (&S0)[pc::D]) { return pc::jit_eval(P, R, a, g, live, Bm, S0" << walk_arg(spec) << "); });\n";
  else
    o << "  pc::price_tiles<pc::D, " << (kind & kJitPriceWrite ? "true" : "false") << ">(a, [&](const uint4 *P, const float *,\n"
      << "      float2 *R, const pc::Rng2 &g, bool live0, bool live1, const float (&Bm)[pc::D * pc::D],\n"
      << "      const float (&S0)[pc::D]) { return pc::jit_eval(P, R, a, g, live0, live1, Bm, S0" << walk_arg(spec) << "); });\n";
  o << "}\n";
  return o.str();
}

pc_status nvrtc_fail(nvrtcResult r, nvrtcProgram prog, const char *what) {
  std::string msg = std::string(what) + ": " + nvrtcGetErrorString(r);
  size_t n = 0;
  if (prog && nvrtcGetProgramLogSize(prog, &n) == NVRTC_SUCCESS && n > 1) {
    std::string log(n, '\0');
    nvrtcGetProgramLog(prog, &log[0]);
    msg += "\n" + log.substr(0, 4000);
  }
  return fail(PC_ECUDA, msg);
}

// NVRTC: the generated source and the embedded device headers to a cubin
// for `arch` (e.g. "sm_103a").
pc_status to_cubin(const Program &p, const JitSpec &spec, const std::string &arch, std::vector<char> &cubin) {
  const std::string src = generate(p, spec);
  nvrtcProgram prog = nullptr;
  nvrtcResult r = nvrtcCreateProgram(&prog, src.c_str(), "pc_jit.cu", kJitHeaderCount, kJitHeaderSrcs,
                                     kJitHeaderNames);
  if (r != NVRTC_SUCCESS) return nvrtc_fail(r, nullptr, "run-time compiler");
  const std::string a = "-arch=" + arch;
  const std::string bound = "-DPC_MIN_BLOCKS=" + std::to_string(spec.min_blocks > 0 ? spec.min_blocks : kJitMinBlocks);
  const char *opts[] = {a.c_str(), "-std=c++17", "-default-device", "-DPC_JIT", bound.c_str(), "-DPC_ONE_PHI"};
  r = nvrtcCompileProgram(prog, spec.one_phi ? 6 : 5, opts);
  if (r != NVRTC_SUCCESS) {
    pc_status s = nvrtc_fail(r, prog, "run-time compilation");
    nvrtcDestroyProgram(&prog);
    return s;
  }
  size_t n = 0;
  r = nvrtcGetCUBINSize(prog, &n);
  cubin.assign(n, 0);
  if (r == NVRTC_SUCCESS) r = nvrtcGetCUBIN(prog, cubin.data());
  nvrtcDestroyProgram(&prog);
  if (r != NVRTC_SUCCESS) return nvrtc_fail(r, nullptr, "cubin");
  return PC_OK;
}

const char *jit_entry_name(int kind) {
  return kind >= kJitAdjoint ? "pc_jit_adjoint" : kind >= kJitGreeks ? "pc_jit_greeks"
         : kind >= kJitCv ? "pc_jit_cv" : "pc_jit_price";
}

pc_status compile(const Program &p, const JitSpec &spec, int device, cudaLibrary_t &lib, cudaKernel_t &kern) {
  cudaDeviceProp prop{};
  CU(cudaGetDeviceProperties(&prop, device), "device properties");
  std::vector<char> cubin;
  pc_status s = to_cubin(p, spec, "sm_" + std::to_string(prop.major) + std::to_string(prop.minor) + "a", cubin);
  if (s != PC_OK) return s;
  CU(cudaLibraryLoadData(&lib, cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0), "module load");
  cudaError_t e = cudaLibraryGetKernel(&kern, lib, jit_entry_name(spec.kind));
  if (e != cudaSuccess) {
    cudaLibraryUnload(lib);
    lib = nullptr;
    kern = nullptr;
    return cuda_fail(e, "kernel lookup");
  }
  return PC_OK;
}

}  // namespace

namespace pc {

bool jit_eligible(const pc_contract *k) { return k->prog.code.size() <= size_t(PC_JIT_MAX_INSNS); }

bool adjoint_jit_eligible(const pc_contract *k) {
  return jit_eligible(k) && date_sites(k->prog) <= kAdjointDateSites;
}

JitSpec jit_spec(const pc_contract *k, const PriceArgs &a, int kind, int min_blocks, const std::vector<int32_t> &walk) {
  JitSpec sp;
  sp.d = a.m.d;
  sp.kind = kind;
  sp.min_blocks = min_blocks;
  sp.walk = walk;
  sp.one_phi = one_phi(a.path_offset, a.n_tiles);
  // constants by value, unless an out-of-line date generator takes them by reference
  if (kind >= kJitCv || !outlined_dates(k->prog)) {
    sp.lay = {a.lay.stack, a.lay.off_bstack, a.lay.off_cache, a.lay.off_win, a.lay.off_xwin, a.lay.words, a.lay.win, a.lay.ids};
    if (walk.empty()) {
      // the general kernel serves every model: what follows the bridge stack
      // (its depth is the grid's) and the window's size come from the
      // arguments, but for a window of one date
      for (int i : {2, 3, 4, 5}) sp.lay[size_t(i)] = -1;
      if (a.lay.win > 1) sp.lay[6] = -1;
    }
  }
  if (!walk.empty()) sp.grid = {a.m.n, a.m.n_hist, a.m.t_now};
  return sp;
}

pc_status jit_pair_kernel(const pc_contract *k, pc_contract::Window *w, const PriceArgs &a, int kind, int min_blocks,
                          const std::vector<int32_t> &walk, cudaKernel_t &out) {
  const bool phi = one_phi(a.path_offset, a.n_tiles);
  for (const pc_contract::Window::Kernel &e : w->kernels)
    if (e.kind == kind && e.min_blocks == min_blocks && e.words == a.lay.words && e.one_phi == phi) {
      out = e.kernel;
      return PC_OK;
    }
  const pc_status s = jit_kernel(k, jit_spec(k, a, kind, min_blocks, walk), out);
  if (s == PC_OK) w->kernels.push_back({kind, min_blocks, a.lay.words, phi, out});
  return s;
}

bool walk_jit_eligible(const Program &p) {
  std::vector<int> sp_at;
  return date_sites(p) <= 2 || (date_sites(p) <= kSharedDateSites && stack_depths(p, sp_at));
}

namespace {
// The program's words: code, then pool bits.
std::vector<uint32_t> program_words(const Program &p) {
  std::vector<uint32_t> words;
  words.reserve(p.code.size() * 4 + p.pool.size());
  for (const XInsn &I : p.code) {
    words.push_back(I.opa);
    words.push_back(I.b);
    words.push_back(I.c);
    words.push_back(I.e);
  }
  for (float f : p.pool) {
    uint32_t u;
    std::memcpy(&u, &f, 4);
    words.push_back(u);
  }
  return words;
}
uint64_t words_hash(const std::vector<uint32_t> &words) {
  uint64_t h = 1469598103934665603ull;  // FNV-1a
  for (uint32_t w : words)
    for (int b = 0; b < 4; ++b) h = (h ^ ((w >> (8 * b)) & 0xffu)) * 1099511628211ull;
  return h;
}
// The cached kernel of these words and this spec (jit_mu held); null if none.
cudaKernel_t cached(pc_ctx *c, uint64_t h, const std::vector<uint32_t> &words, const JitSpec &spec) {
  auto range = c->jit_cache.equal_range(h);
  for (auto it = range.first; it != range.second; ++it)
    if (it->second.spec == spec && it->second.program == words) return it->second.kernel;
  return nullptr;
}
}  // namespace

bool admit_walk(pc_ctx *c, const Program &p, const ModelHost &H, const std::vector<int32_t> &walk) {
  std::vector<int32_t> key = {H.d, H.n, H.n_hist, H.t_now};
  key.insert(key.end(), walk.begin(), walk.end());
  const uint64_t h = words_hash(program_words(p));
  std::lock_guard<std::mutex> g(c->jit_mu);
  auto &known = c->jit_walks[h];
  if (std::find(known.begin(), known.end(), key) != known.end()) return true;
  if (known.size() >= kWalksPerProgram) return false;
  known.push_back(std::move(key));
  return true;
}

pc_status jit_kernel(const pc_contract *k, const JitSpec &spec, cudaKernel_t &out) {
  JitEntry E;
  E.program = program_words(k->prog);
  E.spec = spec;
  const uint64_t h = words_hash(E.program);
  pc_ctx *c = k->ctx;
  std::lock_guard<std::mutex> g(c->jit_mu);
  out = cached(c, h, E.program, spec);
  if (out) return PC_OK;
  pc_status s = compile(k->prog, spec, c->device, E.lib, E.kernel);
  if (s != PC_OK) return s;
  out = E.kernel;
  c->jit_cache.emplace(h, std::move(E));
  return PC_OK;
}

pc_status jit_compile_many(pc_ctx *c, const std::vector<JitRequest> &reqs) {
  // the requests not yet in the context's cache (each once)
  struct Miss {
    const JitRequest *r;
    std::vector<uint32_t> words;
    uint64_t h;
    std::vector<char> cubin;
    pc_status s = PC_OK;
  };
  std::vector<Miss> miss;
  {
    std::lock_guard<std::mutex> g(c->jit_mu);
    for (const JitRequest &r : reqs) {
      Miss m;
      m.r = &r;
      m.words = program_words(r.k->prog);
      m.h = words_hash(m.words);
      bool have = cached(c, m.h, m.words, r.spec) != nullptr;
      for (const Miss &o : miss) have = have || (o.h == m.h && o.r->spec == r.spec && o.words == m.words);
      if (!have) miss.push_back(std::move(m));
    }
  }
  if (miss.empty()) return PC_OK;
  cudaDeviceProp prop{};
  CU(cudaGetDeviceProperties(&prop, c->device), "device properties");
  const std::string arch = "sm_" + std::to_string(prop.major) + std::to_string(prop.minor) + "a";
  // NVRTC on the host's cores, one program per thread at a time
  std::atomic<size_t> next{0};
  auto work = [&]() {
    for (size_t i = next++; i < miss.size(); i = next++) {
      const JitRequest &r = *miss[i].r;
      miss[i].s = to_cubin(r.k->prog, r.spec, arch, miss[i].cubin);
    }
  };
  const unsigned hw = std::max(1u, std::thread::hardware_concurrency());
  const size_t nt = std::min<size_t>(miss.size(), std::min<unsigned>(hw, 32u));
  std::vector<std::thread> pool;
  for (size_t t = 1; t < nt; ++t) pool.emplace_back(work);
  work();
  for (std::thread &t : pool) t.join();
  std::lock_guard<std::mutex> g(c->jit_mu);
  for (Miss &m : miss) {
    if (m.s != PC_OK) return m.s;
    JitEntry E;
    E.program = m.words;
    E.spec = m.r->spec;
    CU(cudaLibraryLoadData(&E.lib, m.cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0), "module load");
    cudaError_t e = cudaLibraryGetKernel(&E.kernel, E.lib, jit_entry_name(E.spec.kind));
    if (e != cudaSuccess) {
      cudaLibraryUnload(E.lib);
      return cuda_fail(e, "kernel lookup");
    }
    c->jit_cache.emplace(m.h, std::move(E));
  }
  return PC_OK;
}

void jit_release(pc_ctx *c) {
  std::lock_guard<std::mutex> g(c->jit_mu);
  for (auto &kv : c->jit_cache)
    if (kv.second.lib) cudaLibraryUnload(kv.second.lib);
  c->jit_cache.clear();
}

}  // namespace pc

extern "C" pc_status pc_debug_jit_compile(const uint32_t *bytecode, size_t n_words, const double *consts,
                                          size_t n_consts, const int32_t *tparams, size_t n_params,
                                          int32_t p1, int32_t p2, int32_t d, int32_t kind,
                                          size_t *cubin_bytes) {
  if (!cubin_bytes) return fail(PC_EINVAL, "null output");
  if (d < 1 || d > PC_MAX_UNDERLYINGS) return fail(PC_EINVAL, "d must be 1..4");
  const int cvm = (kind - kJitCv) & 7;  // mode bits, with or without kCvWinRegs
  const bool cv_kind = kind >= kJitCv && kind < kJitCv + 16 && cvm != kCvWrite && cvm != (kCvWrite | kCvPilot) &&
                       cvm != (kCvWrite | kCvPilot | kCvGamma);
  const bool greeks_kind = kind == kJitGreeks || kind == kJitGreeks + 1 || kind == kJitAdjoint ||
                           kind == kJitAdjoint + 1;
  const bool price_kind = kind >= 0 && kind <= (kJitPriceWrite | kJitHbm | kJitWinRegs | kJitPairs2) &&
                          (!(kind & kJitPairs2) || (kind & (kJitWinRegs | kJitHbm)) == kJitWinRegs);
  if (!price_kind && !cv_kind && !greeks_kind)
    return fail(PC_EINVAL, "unknown kernel kind");
  if (cv_kind && d > kCvMaxD) return fail(PC_EINVAL, "control-variate kernels take d <= 3");
  Program p;
  std::string err;
  pc_status s = compile_program(bytecode, n_words, consts, n_consts, tparams, n_params, p1, p2, true, p, err);
  if (s != PC_OK) return fail(s, err);
  std::vector<char> cubin;
  s = to_cubin(p, JitSpec{d, kind}, "sm_103a", cubin);
  if (s != PC_OK) return s;
  *cubin_bytes = cubin.size();
  return PC_OK;
}

extern "C" pc_status pc_debug_jit_source(const uint32_t *bytecode, size_t n_words, const double *consts,
                                         size_t n_consts, const int32_t *tparams, size_t n_params,
                                         int32_t p1, int32_t p2, int32_t d, int32_t kind, char *out,
                                         size_t cap, size_t *len) {
  if (!len) return fail(PC_EINVAL, "null output");
  if (d < 1 || d > PC_MAX_UNDERLYINGS) return fail(PC_EINVAL, "d must be 1..4");
  const bool known = (kind >= 0 && kind <= (kJitPriceWrite | kJitHbm | kJitWinRegs | kJitPairs2) &&
                      (!(kind & kJitPairs2) || (kind & (kJitWinRegs | kJitHbm)) == kJitWinRegs)) ||
                     (kind >= kJitCv && kind < kJitCv + 16) ||
                     kind == kJitGreeks || kind == kJitGreeks + 1 || kind == kJitAdjoint || kind == kJitAdjoint + 1;
  if (!known) return fail(PC_EINVAL, "unknown kernel kind");
  Program p;
  std::string err;
  pc_status s = compile_program(bytecode, n_words, consts, n_consts, tparams, n_params, p1, p2, true, p, err);
  if (s != PC_OK) return fail(s, err);
  const std::string src = generate(p, JitSpec{d, kind});
  *len = src.size();
  if (out && cap > src.size()) std::memcpy(out, src.c_str(), src.size() + 1);
  return PC_OK;
}
