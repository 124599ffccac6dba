// Translation of a plan's stream into compact records (compact.h).
#include "compact.h"

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>

namespace ndvm {
namespace {

// NDVM_COMPACT=0 keeps every tape on the general interpreter (a tuning knob).
bool compact_enabled() {
  const char* e = std::getenv("NDVM_COMPACT");
  return !(e && e[0] == '0');
}

uint32_t slot(int32_t ref) { return ref == -1 ? kCNone : (uint32_t)ref_index(ref) * kCSlotUnit; }

// Whether a record reads the slot at offset s (a constant's load that nothing reads
// before the slot is written again is left out).
bool reads(const CRec& c, uint32_t s) {
  auto range = [&] { return s >= c.w[1] && s < c.w[1] + c.w[2] * kCSlotUnit; };
  switch (c.w[0] & 0xff) {
    case C_ARITH: return c.w[2] == s || c.w[3] == s || c.w[4] == s;
    case C_LOOP: return c.w[5] == s;
    case C_ZERO: return false;
    case C_GREDUCE: return range();
    case C_LOSS: case C_GRAD: return c.w[1] == s;
    case C_DIV: return c.w[2] == s || c.w[3] == s || c.w[4] == s;
    case C_POW: case C_CMP: return c.w[2] == s || c.w[3] == s;
    case C_RCP: case C_EXP: case C_LOG: case C_TANH: case C_SQRT: case C_ABS: case C_SIN: case C_COS: case C_POWI:
      return c.w[2] == s;
    case C_SELECT: return c.w[2] == s || c.w[3] == s || c.w[4] == s;
    case C_LOADC: case C_LOADP: case C_LOADO: case C_LOADS: case C_OBS: case C_FETCH: case C_SEED: case C_END:
    case C_ENDLOOP: case C_CHUNK:
      return false;
    default:  // reverse rules: the adjoint, the targets (accumulated into) and the operands
      for (int k = 1; k <= 7; k++)
        if (c.w[k] == s) return true;
      return false;
  }
}

// The records of p.code; empty when an instruction has no compact form.
std::vector<CRec> translate(const Plan& p, const std::vector<double>& consts, int64_t* max_points) {
  const std::vector<CRec> none;
  std::vector<double> pool = consts;
  pool.insert(pool.end(), p.extra_consts.begin(), p.extra_consts.end());
  const int32_t valid_slot = p.n_slots + kCSlotValid;
  const uint32_t valid = (uint32_t)valid_slot * kCSlotUnit;
  const uint32_t one = (uint32_t)(p.n_slots + kCSlotOne) * kCSlotUnit;
  const uint32_t mzero = (uint32_t)(p.n_slots + kCSlotMinusZero) * kCSlotUnit;
  std::vector<CRec> code;
  auto rec = [&](uint32_t op, uint32_t w1 = 0, uint32_t w2 = 0) -> CRec& {
    CRec c;
    c.w[0] = op;
    c.w[1] = w1;
    c.w[2] = w2;
    code.push_back(c);
    return code.back();
  };
  auto loadc = [&](uint32_t dst, double v) {
    const float f = (float)v;
    uint64_t b;
    uint32_t bf;
    std::memcpy(&b, &v, 8);
    std::memcpy(&bf, &f, 4);
    CRec& c = rec(C_LOADC, dst, (uint32_t)b);
    c.w[3] = (uint32_t)(b >> 32);
    c.w[4] = bf;
  };
  loadc(one, 1.0);
  loadc(mzero, -0.0);
  auto load = [&](int32_t dst, int32_t ref) {  // false: not a kind a scalar stream loads here
    const int32_t idx = ref_index(ref);
    switch (ref_kind(ref)) {
      case RK_CONST: loadc(slot(dst), pool[(size_t)idx]); return true;
      case RK_PARAM: rec(C_LOADP, slot(dst), (uint32_t)idx); return true;
      case RK_OBS: rec(C_LOADO, slot(dst), (uint32_t)idx); return true;
      case RK_SAVE: rec(C_LOADS, slot(dst), (uint32_t)idx); return true;
      default: return false;
    }
  };
  // copies gathered from consecutive fetch instructions into records of kCCopies
  std::vector<std::pair<uint32_t, uint32_t>> copies;
  auto flush = [&](uint32_t op, uint32_t last_flags) {
    size_t e = 0;
    do {
      const size_t m = std::min<size_t>(kCCopies, copies.size() - e);
      CRec& c = rec(op | ((uint32_t)m << kCCountShift));
      for (size_t q = 0; q < m; q++) {
        c.w[1 + 2 * q] = copies[e + q].first;
        c.w[2 + 2 * q] = copies[e + q].second;
      }
      e += m;
      if (e >= copies.size()) c.w[0] |= last_flags;
    } while (e < copies.size());
    copies.clear();
  };
  int loop_pc = -1;           // the open C_LOOP record
  int32_t seed = -1;          // slot of a seed set before the loop being translated
  int32_t pending_seed = -1;  // slot of a seed set just before a loop
  for (size_t pc = 0; pc < p.code.size(); pc++) {
    const DInst& d = p.code[pc];
    const int32_t* f = d.f;
    const uint32_t fa = (d.flags & 1) ? kCFirstA : 0, fb = (d.flags & 2) ? kCFirstB : 0;
    auto fwd = [&](uint32_t op) -> CRec& {  // result, operands, save
      CRec& c = rec(op, slot(f[0]), slot(f[1]));
      c.w[3] = slot(f[2]);
      c.w[5] = c.w[6] = kCNone;
      c.w[7] = (uint32_t)f[3];
      if (f[3] >= 0) c.w[0] |= kCSave;
      return c;
    };
    auto arith = [&](int32_t dst, int32_t x, bool neg, int32_t y, int32_t z, int32_t save, uint32_t flags) {
      CRec& c = rec(C_ARITH | flags | (neg ? kCNeg : 0), slot(dst), slot(x));
      c.w[3] = y != -1 ? slot(y) : one;
      c.w[4] = z != -1 ? slot(z) : mzero;
      c.w[0] |= (y != -1 ? kCHasB : 0) | (z != -1 ? kCHasC : 0);
      c.w[7] = (uint32_t)save;
      if (save >= 0) c.w[0] |= kCSave;
    };
    auto rev = [&](uint32_t op) -> CRec& {
      CRec& c = rec(op | fa | fb, slot(f[0]), slot(f[1]));
      c.w[3] = slot(f[2]);
      c.w[4] = slot(f[3]);
      c.w[5] = slot(f[4]);
      c.w[6] = slot(f[5]);
      c.w[7] = slot(f[6]);
      return c;
    };
    switch (d.op) {
      case D_FMA: {
        const bool gate = !(d.flags & kFmaNoGate);
        if (gate && f[4] != f[1]) return none;
        const int32_t y = (d.flags & kFmaUnitB) ? -1 : f[2], z = (d.flags & kFmaZeroC) ? -1 : f[3];
        if (d.flags & kFmaAcc) {
          // the body's value added once per point: by a factor of the point's validity
          if (loop_pc < 0) return none;
          CRec& c = rec(C_ARITH | kCGate | kCHasB | kCHasC, slot(f[0]), valid);
          c.w[3] = slot(f[1]);
          c.w[4] = slot(f[3]);
          c.w[7] = (uint32_t)-1;
          break;
        }
        arith(f[0], f[1], d.flags & 1, y, z, f[5], gate ? kCGate : 0);
        break;
      }
      // (the general forward forms: derive plans; exact, as in the fused form)
      case D_ADD: arith(f[0], f[1], false, -1, f[2], f[3], 0); break;
      case D_SUB: arith(f[0], f[2], true, -1, f[1], f[3], 0); break;
      case D_MUL: arith(f[0], f[1], false, f[2], -1, f[3], 0); break;
      case D_NEG: arith(f[0], f[1], true, -1, -1, f[3], 0); break;
      case D_DIV: {
        CRec& c = fwd(C_DIV);
        c.w[4] = kCNone;
        c.w[5] = slot(f[4]);
        if (f[5] >= 0) return none;
        break;
      }
      case D_POW: fwd(C_POW); break;
      case D_EXP: fwd(C_EXP); break;
      case D_LOG: fwd(C_LOG); break;
      case D_TANH: fwd(C_TANH); break;
      case D_SQRT: fwd(C_SQRT); break;
      case D_ABS: fwd(C_ABS); break;
      case D_SIN: case D_COS: {
        CRec& c = fwd(d.op == D_SIN ? C_SIN : C_COS);
        c.w[5] = slot(f[4]);
        c.w[6] = (uint32_t)f[5];
        break;
      }
      case D_POWI: fwd(C_POWI).w[6] = (uint32_t)f[7]; break;
      case D_CMP: fwd(C_CMP | ((uint32_t)d.k << kCCountShift)); break;
      case D_SELECT: fwd(C_SELECT).w[4] = slot(f[4]); break;
      case D_ZERO: rec(C_ZERO, slot(f[0]), (uint32_t)f[1]); break;
      case D_LOOP: {
        if (loop_pc >= 0) return none;
        seed = pending_seed;
        CRec& c = rec(C_LOOP, (uint32_t)f[0], (uint32_t)f[1]);
        c.w[3] = (uint32_t)f[2];
        c.w[5] = valid;
        loop_pc = (int)code.size() - 1;
        *max_points = std::max<int64_t>(*max_points, f[0]);
        break;
      }
      case D_ENDLOOP:
        if (loop_pc < 0) return none;
        code[(size_t)loop_pc].w[4] = (uint32_t)code.size();
        rec(C_ENDLOOP);
        // a seed set before the loop is the points' validity inside it
        if (seed != -1)
          for (size_t q = (size_t)loop_pc + 1; q < code.size(); q++) {
            CRec& c = code[q];
            const uint32_t s = slot(seed);
            const uint32_t op = c.w[0] & 0xff;
            if (op == C_ARITH) {
              if (c.w[1] == s) return none;
              for (int k = 2; k <= 4; k++)
                if (c.w[k] == s) c.w[k] = valid;
            } else if (op >= R_DIV && op <= R_DSUM) {
              if (c.w[2] == s || c.w[3] == s) return none;
              if (c.w[1] == s) c.w[1] = valid;
              for (int k = 4; k <= 7; k++)
                if (c.w[k] == s) return none;
            } else if (op != C_ENDLOOP && (c.w[1] == s || reads(c, s))) {
              return none;
            }
          }
        loop_pc = -1;
        seed = -1;
        break;
      case D_SEED:
        if (loop_pc >= 0) {  // inside a loop: 1 at a valid point, 0 elsewhere
          arith(f[0], mkref(RK_SLOT, valid_slot), false, -1, -1, -1, 0);
        } else {
          rec(C_SEED, slot(f[0]));
          bool before_loop = false;  // only loads and other seeds between it and a loop
          for (size_t q = pc + 1; q < p.code.size(); q++) {
            if (p.code[q].op == D_LOOP) before_loop = true;
            if (p.code[q].op != D_LOAD) break;
          }
          pending_seed = before_loop ? f[0] : -1;
        }
        break;
      case D_GREDUCE: rec(C_GREDUCE, slot(f[0]), (uint32_t)f[1]); break;
      case D_LOAD:
        if (loop_pc >= 0 && ref_kind(f[1]) == RK_DOBS) {
          copies.push_back({slot(f[0]), (uint32_t)ref_index(f[1])});
          flush(C_OBS, 0);
          break;
        }
        if (!load(f[0], f[1])) return none;
        break;
      case D_LOSS:
        if (ref_kind(f[0]) == RK_SLOT) {
          rec(C_LOSS, slot(f[0]));
        } else {
          if (!load(mkref(RK_SLOT, valid_slot), f[0])) return none;
          rec(C_LOSS, valid);
        }
        break;
      case D_FETCH: {
        const bool from_obs = d.flags & 32;
        if (from_obs && loop_pc < 0) return none;
        for (int e = 0; e < d.k; e++) copies.push_back({slot(f[2 * e + 1]), (uint32_t)ref_index(f[2 * e])});
        if (from_obs) { flush(C_OBS, 0); break; }
        if (!(d.flags & 3) && pc + 1 < p.code.size() && p.code[pc + 1].op == D_FETCH) break;  // one run of copies
        flush(C_FETCH, ((d.flags & 2) ? kCCommit : 0) | ((d.flags & 1) ? kCWait : 0) |
                           ((uint32_t)((d.flags >> 2) & 7) << kCPendingShift));
        break;
      }
      case B_DIV: rev(R_DIV); break;
      case B_POW: rev(R_POW); break;
      case B_TANH: if (f[1] != -1) rev(R_TANH); break;
      case B_LOG: if (f[1] != -1) rev(R_LOG); break;
      case B_ABS: if (f[1] != -1) rev(R_ABS); break;
      case B_SQRT: if (f[1] != -1) rev(R_SQRT); break;
      case B_POWI: if (f[1] != -1) rev(R_POWI).w[7] = (uint32_t)f[7]; break;
      case B_SELECT: rev(R_SELECT); break;
      case B_DSUM:
        for (int e = 0; e < f[2]; e++) {
          const int32_t* q = &p.args[(size_t)f[1] + 3 * (size_t)e];
          CRec& c = rec(R_DSUM | (q[1] ? kCFirstA : 0), slot(f[0]), slot(q[0]));
          c.w[3] = kCNone;
          c.w[4] = slot(q[2]);
          c.w[5] = c.w[6] = c.w[7] = kCNone;
        }
        break;
      case B_GRAD: rec(C_GRAD, slot(f[0]), (uint32_t)f[1]); break;
      default: return none;
    }
    if (d.op != D_SEED && d.op != D_LOAD) pending_seed = -1;
  }
  if (loop_pc >= 0 || !copies.empty()) return none;
  rec(C_END);
  // constants that only stood in for an absent operand are not loaded
  std::vector<char> dead(code.size(), 0);
  for (size_t q = 0; q < code.size(); q++) {
    if ((code[q].w[0] & 0xff) != C_LOADC) continue;
    const uint32_t s = code[q].w[1];
    bool used = false;
    for (size_t k = q + 1; k < code.size() && !used; k++) used = reads(code[k], s);
    dead[q] = !used;
  }
  std::vector<uint32_t> newpc(code.size());
  std::vector<CRec> kept;
  for (size_t q = 0; q < code.size(); q++) {
    newpc[q] = (uint32_t)kept.size();
    if (!dead[q]) kept.push_back(code[q]);
  }
  for (CRec& c : kept)
    if ((c.w[0] & 0xff) == C_LOOP) c.w[4] = newpc[c.w[4]];
  return kept;
}

// The slot that a record writes, when it writes one value (kCNone otherwise); all = false when it
// may write others too.
uint32_t writes(const CRec& c, bool* all) {
  const uint32_t op = c.w[0] & 0xff;
  *all = true;
  if (op == C_ARITH || op == C_LOADC || op == C_LOADP || op == C_LOADO || op == C_LOADS || op == C_SEED || op == C_RCP) return c.w[1];
  if (op == C_LOSS || op == C_GRAD || op == C_END || op == C_ENDLOOP) return kCNone;
  *all = false;
  return kCNone;
}

// Divisions by one value that the whole stream divides by more than once share its
// reciprocal: 1 / b is computed where b is (once per lane when b is a lane's value and the
// division a point's), and each division takes the product and the correction step that
// follow the reciprocal anyway (3 FP64 instructions of 7).  b's slot must have one writer,
// outside loops, ahead of the divisions, so that it holds b wherever it is read.
void share_reciprocals(std::vector<CRec>& code, int32_t* n_slots) {
  struct Use { int writers = 0, writer = -1, divisions = 0; bool in_loop = false; };
  std::map<uint32_t, Use> use;
  bool loop = false;
  auto write = [&](uint32_t s, int pc) {
    Use& u = use[s];
    u.writers++;
    u.writer = pc;
    u.in_loop |= loop;
  };
  for (int pc = 0; pc < (int)code.size(); pc++) {
    const CRec& c = code[(size_t)pc];
    const uint32_t op = c.w[0] & 0xff;
    if (op == C_LOOP) { loop = true; write(c.w[5], pc); }
    if (op == C_ENDLOOP) loop = false;
    bool one;
    const uint32_t s = writes(c, &one);
    if (s != kCNone) write(s, pc);
    if (one || op == C_LOOP || op == C_ENDLOOP) continue;
    if (op == C_ZERO || op == C_GREDUCE) {
      for (uint32_t e = 0; e < c.w[2]; e++) write(c.w[1] + e * kCSlotUnit, pc);
    } else if (op == C_FETCH || op == C_OBS) {
      for (int e = 0; e < (int)((c.w[0] >> kCCountShift) & 7); e++) write(c.w[1 + 2 * e], pc);
    } else if (op >= R_DIV && op <= R_DSUM) {
      for (int k = 2; k <= 3; k++) if (c.w[k] != kCNone) write(c.w[k], pc);
    } else {  // forward functions: the result and an auxiliary value
      write(c.w[1], pc);
      if (op != C_SELECT && c.w[5] != kCNone) write(c.w[5], pc);
    }
  }
  for (const CRec& c : code) {
    const uint32_t op = c.w[0] & 0xff;
    if (op == C_DIV) use[c.w[3]].divisions++;
    if (op == R_DIV) use[c.w[5]].divisions++;
  }
  // (a division inside a loop runs once per point, so one is enough there)
  std::map<int, uint32_t> make;      // writer pc -> divisor's slot
  std::map<uint32_t, uint32_t> rcp;  // divisor's slot -> reciprocal's
  loop = false;
  for (int pc = 0; pc < (int)code.size(); pc++) {
    const CRec& c = code[(size_t)pc];
    const uint32_t op = c.w[0] & 0xff;
    if (op == C_LOOP) loop = true;
    if (op == C_ENDLOOP) loop = false;
    if (op != C_DIV) continue;
    const Use& u = use[c.w[3]];
    if (u.writers != 1 || u.in_loop || u.writer >= pc || (u.divisions < 2 && !loop) || rcp.count(c.w[3])) continue;
    if ((int)rcp.size() >= kCMaxReciprocals) break;
    make[u.writer] = c.w[3];
    rcp[c.w[3]] = (uint32_t)(*n_slots)++ * kCSlotUnit;
  }
  if (rcp.empty()) return;
  std::map<uint32_t, uint32_t> aux;  // a division's own reciprocal slot -> the shared one
  std::vector<CRec> out;
  std::vector<uint32_t> newpc(code.size());
  for (int pc = 0; pc < (int)code.size(); pc++) {
    CRec c = code[(size_t)pc];
    const uint32_t op = c.w[0] & 0xff;
    newpc[(size_t)pc] = (uint32_t)out.size();
    if (op == C_DIV && rcp.count(c.w[3])) {
      c.w[4] = rcp[c.w[3]];
      c.w[5] = kCNone;
    }
    if (op == R_DIV && rcp.count(c.w[5])) c.w[7] = rcp[c.w[5]];
    out.push_back(c);
    if (make.count(pc)) {
      CRec r;
      r.w[0] = C_RCP;
      r.w[1] = rcp[make[pc]];
      r.w[2] = make[pc];
      out.push_back(r);
    }
  }
  for (CRec& c : out)
    if ((c.w[0] & 0xff) == C_LOOP) c.w[4] = newpc[c.w[4]];
  code.swap(out);
}

// A long stream's chunks: the last record of each says so.
void mark_chunks(std::vector<CRec>& code) {
  std::vector<CRec> out;
  CRec mark;
  mark.w[0] = C_CHUNK;
  for (const CRec& c : code) {
    if (out.size() % kCChunk == kCChunk - 1) out.push_back(mark);
    out.push_back(c);
  }
  code.swap(out);
}

}  // namespace

void compact_plan(Plan& p, const std::vector<double>& consts) {
  for (Plan& d : p.derive) compact_plan(d, consts);
  p.compact.clear();
  p.compact_slots = p.n_slots + kCExtraSlots;
  p.compact_points = 0;
  if (!compact_enabled()) return;
  std::vector<CRec> code = translate(p, consts, &p.compact_points);
  if (code.empty()) return;
  share_reciprocals(code, &p.compact_slots);
  if (p.compact_points == 0 && code.size() > kCResident) mark_chunks(code);
  for (const CRec& c : code) p.compact.insert(p.compact.end(), c.w, c.w + kCompactWords);
}

}  // namespace ndvm
