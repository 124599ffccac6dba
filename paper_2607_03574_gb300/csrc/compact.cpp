// Translation of a plan's stream into compact records (compact.h).
#include "compact.h"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <map>

#include "cost.h"

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
template <typename R>
bool reads(const R& c, uint32_t s) {
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

// The factor m of e / cols = (e m) >> 20 for the elements e of a matrix of up to 64 x 64.
uint32_t row_of(int cols) { return ((1u << 20) + (uint32_t)cols - 1) / (uint32_t)cols; }

// What a matrix stream holds besides its records: the constant matrices its operands name, the
// lists of their nonzero elements, and the staged operands -- workspace values and observations,
// copied into slots of their own a few records before they are used.
struct Matrices {
  struct Stage {
    bool from_obs;
    int32_t src;
    int width;
    int use_first, use_last;                   // records that read it
    std::vector<std::pair<int, int>> patches;  // (record, word)
    int fetch_at = 0, slot = 0;
  };
  std::vector<double> consts;
  std::vector<int32_t> lists;
  std::vector<Stage> stages;
  int rev_begin = -1;  // first record of the reverse sweep
  int temps = 1;       // slots for parameters that are operands: a record's two have one each

  int constants(const std::vector<double>& pool, int32_t idx, int width) {
    auto it = runs_.find({idx, width});
    if (it != runs_.end()) return it->second;
    const int at = (int)consts.size();
    consts.insert(consts.end(), pool.begin() + idx, pool.begin() + idx + width);
    runs_[{idx, width}] = at;
    return at;
  }
  int list(const std::vector<int32_t>& l) {
    auto it = known_.find(l);
    if (it != known_.end()) return it->second;
    const int at = (int)lists.size();
    lists.insert(lists.end(), l.begin(), l.end());
    known_[l] = at;
    return at;
  }
  // the copy of a run of source elements that record `rec` reads; one made for a record
  // shortly before serves again
  int stage(bool from_obs, int32_t src, int width, int rec) {
    for (int k = (int)stages.size() - 1; k >= 0 && k >= (int)stages.size() - 8; k--) {
      const Stage& s = stages[(size_t)k];
      if (s.from_obs == from_obs && s.src == src && s.width == width && s.use_last >= rec - 2 * kMAhead) return k;
    }
    Stage s;
    s.from_obs = from_obs;
    s.src = src;
    s.width = width;
    s.use_first = s.use_last = rec;
    stages.push_back(s);
    return (int)stages.size() - 1;
  }
  void use(int k, int rec, int word) {
    Stage& s = stages[(size_t)k];
    if (s.patches.empty()) s.use_first = rec;
    s.use_last = rec;
    s.patches.push_back({rec, word});
  }

 private:
  std::map<std::pair<int32_t, int>, int> runs_;
  std::map<std::vector<int32_t>, int> known_;
};

// The records of p.code (the first kCompactWords words of each for a scalar stream); empty when an
// instruction has no compact form.  `mx`: matrix instructions too.
std::vector<MRec> translate(const Plan& p, const std::vector<double>& consts, int64_t* max_points, Matrices* mx) {
  const std::vector<MRec> none;
  std::vector<double> pool = consts;
  pool.insert(pool.end(), p.extra_consts.begin(), p.extra_consts.end());
  const int32_t valid_slot = p.n_slots + kCSlotValid;
  const uint32_t valid = (uint32_t)valid_slot * kCSlotUnit;
  const uint32_t one = (uint32_t)(p.n_slots + kCSlotOne) * kCSlotUnit;
  const uint32_t mzero = (uint32_t)(p.n_slots + kCSlotMinusZero) * kCSlotUnit;
  std::vector<MRec> code;
  auto rec = [&](uint32_t op, uint32_t w1 = 0, uint32_t w2 = 0) -> MRec& {
    MRec c;
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
    MRec& c = rec(C_LOADC, dst, (uint32_t)b);
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
      MRec& c = rec(op | ((uint32_t)m << kCCountShift));
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
  std::vector<int32_t> seeds;  // slots of the seeds set since the last loop
  struct Known { uint32_t op; int nz, list; uint32_t flags; };
  std::map<std::vector<int32_t>, Known> products;  // by a product's operands and shape
  int32_t last_product = -1;  // slot of the product that the last record computes
  int last_product_pc = -1;
  std::pair<int32_t, int> last_in[2];  // its operands and their elements
  auto pool_at = [&](int32_t idx, int e) { return pool[(size_t)idx + (size_t)e]; };
  for (size_t pc = 0; pc < p.code.size(); pc++) {
    const DInst& d = p.code[pc];
    const int32_t* f = d.f;
    const uint32_t fa = (d.flags & 1) ? kCFirstA : 0, fb = (d.flags & 2) ? kCFirstB : 0;
    auto fwd = [&](uint32_t op) -> MRec& {  // result, operands, save
      MRec& c = rec(op, slot(f[0]), slot(f[1]));
      c.w[3] = slot(f[2]);
      c.w[5] = c.w[6] = kCNone;
      c.w[7] = (uint32_t)f[3];
      if (f[3] >= 0) c.w[0] |= kCSave;
      return c;
    };
    auto arith = [&](int32_t dst, int32_t x, bool neg, int32_t y, int32_t z, int32_t save, uint32_t flags) {
      MRec& c = rec(C_ARITH | flags | (neg ? kCNeg : 0), slot(dst), slot(x));
      c.w[3] = y != -1 ? slot(y) : one;
      c.w[4] = z != -1 ? slot(z) : mzero;
      c.w[0] |= (y != -1 ? kCHasB : 0) | (z != -1 ? kCHasC : 0);
      c.w[7] = (uint32_t)save;
      if (save >= 0) c.w[0] |= kCSave;
    };
    auto rev = [&](uint32_t op) -> MRec& {
      MRec& c = rec(op | fa | fb, slot(f[0]), slot(f[1]));
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
          MRec& c = rec(C_ARITH | kCGate | kCHasB | kCHasC, slot(f[0]), valid);
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
        MRec& c = fwd(C_DIV);
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
        MRec& c = fwd(d.op == D_SIN ? C_SIN : C_COS);
        c.w[5] = slot(f[4]);
        c.w[6] = (uint32_t)f[5];
        break;
      }
      case D_POWI: fwd(C_POWI).w[6] = (uint32_t)f[7]; break;
      case D_CMP: fwd(C_CMP | ((uint32_t)d.k << kCCountShift)); break;
      case D_SELECT: fwd(C_SELECT).w[4] = slot(f[4]); break;
      case D_ZERO: rec(C_ZERO, slot(f[0]), (uint32_t)f[1]); break;
      case D_LOOP: {
        if (loop_pc >= 0 || mx) return none;
        seed = pending_seed;
        // (a seed that the loop's body may read and that is not the points' validity there would
        // count the points past the last one)
        for (int32_t s : seeds)
          if (s != seed) return none;
        MRec& c = rec(C_LOOP, (uint32_t)f[0], (uint32_t)f[1]);
        c.w[3] = (uint32_t)f[2];
        for (const DeriveInfo& di : p.derive_info)
          if (f[1] == 1 && f[2] == p.n_obs_min + di.offset) c.w[0] |= kCExt;
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
            MRec& c = code[q];
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
        seeds.clear();
        break;
      case D_SEED:
        if (mx && mx->rev_begin < 0) mx->rev_begin = (int)code.size();
        if (loop_pc >= 0) {  // inside a loop: 1 at a valid point, 0 elsewhere
          arith(f[0], mkref(RK_SLOT, valid_slot), false, -1, -1, -1, 0);
        } else {
          rec(C_SEED, slot(f[0]));
          seeds.push_back(f[0]);
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
          MRec& c = rec(R_DSUM | (q[1] ? kCFirstA : 0), slot(f[0]), slot(q[0]));
          c.w[3] = kCNone;
          c.w[4] = slot(q[2]);
          c.w[5] = c.w[6] = c.w[7] = kCNone;
        }
        break;
      case B_GRAD: rec(C_GRAD, slot(f[0]), (uint32_t)f[1]); break;
      default: {
        // ------------------------------------------------------------- matrices
        if (!mx) return none;
        if (d.op >= B_ADD && mx->rev_begin < 0) mx->rev_begin = (int)code.size();
        // operand `field` of the record about to be appended: a slot, an index into the stream's
        // constants (flag set), or a staged copy (patched when its slots are known)
        uint32_t flags = 0;
        std::vector<std::pair<int, int>> staged;  // (field, stage)
        bool ok = true;
        auto operand = [&](int32_t ref, int width, int field, uint32_t const_flag) -> uint32_t {
          switch (ref_kind(ref)) {
            case RK_SLOT: return slot(ref);
            case RK_CONST:
              if (!const_flag) break;
              flags |= const_flag;
              return (uint32_t)mx->constants(pool, ref_index(ref), width);
            case RK_PARAM: {
              if (width != 1) break;
              const int second = field & 1;  // (of the fields 2 and 3, or 5 and 6)
              mx->temps = std::max(mx->temps, 1 + second);
              const int32_t tmp = p.n_slots + kCExtraSlots + second;
              load(mkref(RK_SLOT, tmp), ref);
              return slot(tmp);
            }
            case RK_SAVE: case RK_OBS:
              staged.push_back({field, mx->stage(ref_kind(ref) == RK_OBS, ref_index(ref), width, (int)code.size())});
              return 0;
            default: break;
          }
          ok = false;
          return 0;
        };
        auto append = [&](uint32_t op) -> MRec& {
          for (const auto& s : staged) mx->use(s.second, (int)code.size(), s.first);
          staged.clear();
          MRec& c = rec(op | flags);
          c.w[7] = (uint32_t)-1;
          flags = 0;
          return c;
        };
        auto save = [&](MRec& c, int32_t idx) {
          c.w[7] = (uint32_t)idx;
          if (idx >= 0) c.w[0] |= kCSave;
        };
        // element (i, j) of the result = sum over q of X[i xi + q xq] Y[q yq + j yj]
        auto mm = [&](int32_t out, int32_t X, int wx, int xi, int xq, int32_t Y, int wy, int yq, int yj, int rows, int cols,
                      int K, uint32_t more, int gate, int32_t sv) {
          const uint32_t x = operand(X, wx, 2, kMConstX), y = operand(Y, wy, 3, kMConstY);
          int nz = 0, list = 0;
          const bool reverse = more & (kMGateX | kMGateY);
          uint32_t op = (reverse ? M_R : M_F) + (K <= 8 ? (uint32_t)K : 0u);
          if (ok) {
            const bool cx = flags & kMConstX, cy = flags & kMConstY;
            const std::vector<int32_t> key = {cx ? X : -1, cy ? Y : ref_kind(Y) == RK_OBS ? -2 : -1, ref_kind(X) == RK_OBS, xi, xq, yq, yj, rows, cols, K, (int32_t)more};
            auto known = cx || cy ? products.find(key) : products.end();
            if (known != products.end()) {
              op = known->second.op;
              nz = known->second.nz;
              list = known->second.list;
              flags |= known->second.flags;
            } else if (cx || cy) {
              const uint32_t had = flags;
              int best = K;
              for (int side = 0; side < 2; side++) {  // the constant operand's nonzero elements
                // (observations are not checked for infinities: every term)
                if (!(side ? cy : cx) || ref_kind(side ? X : Y) == RK_OBS) continue;
                const int32_t at = ref_index(side ? Y : X);
                const int outer = side ? cols : rows, so = side ? yj : xi, sq = side ? yq : xq;
                bool finite = true, unit = true, odd = false;
                int most = 1;
                for (int o = 0; o < outer; o++) {
                  int m = 0;
                  for (int q = 0; q < K; q++) {
                    const double v = pool_at(at, o * so + q * sq);
                    finite = finite && std::isfinite(v);
                    if (v != 0) { m++; unit = unit && v == 1.0; odd = odd || q % 2 == 1; }
                  }
                  most = std::max(most, m);
                }
                // (both operands constant: an infinity or a NaN in the other one is no stored value that
                // the kernel would have met, and binary32 has more infinities; zeros times them count)
                if (side ? cx : cy) {
                  const int32_t oat = ref_index(side ? X : Y);
                  for (int e = 0; e < (side ? wx : wy); e++) finite = finite && std::isfinite((float)pool_at(oat, e));
                }
                if (!finite || most >= best) continue;
                best = most;
                const bool select = most == 1 && unit && !(more & kMAcc) && !(side ? cx : cy);
                // (sums over more than 8 terms take the even and the odd ones in two chains, as the
                // dense products do: the same roundings whichever kernel a lane runs on)
                const bool chains = K > 8 && odd && !select;
                nz = most + (chains ? 1 : 0);
                std::vector<int32_t> l;
                for (int i = 0; i < rows; i++)
                  for (int j = 0; j < cols; j++) {
                    const size_t end = l.size() + (size_t)nz;
                    const int o = side ? j : i;
                    auto terms = [&](int from, int step) {
                      for (int q = from; q < K; q += step) {
                        if (pool_at(at, o * so + q * sq) == 0) continue;
                        const uint32_t ce = (uint32_t)((side ? y : x) + (uint32_t)(o * so + q * sq));
                        const uint32_t oe = (uint32_t)(side ? i * xi + q * xq : q * yq + j * yj);
                        l.push_back((int32_t)(select ? oe : ce | oe << 16));
                      }
                    };
                    terms(0, chains ? 2 : 1);
                    if (chains) {
                      l.push_back((int32_t)kMSplit);
                      terms(1, 2);
                    }
                    l.resize(end, (int32_t)kCNone);
                  }
                list = mx->list(l);
                op = reverse ? (select ? M_RSELECT : M_RSPARSE) : select ? M_SELECT : M_FSPARSE;
                flags = (flags & ~(kMOtherY | kMChains)) | (side ? 0 : kMOtherY) | (chains ? kMChains : 0);
              }
              // (a variable operand's slots differ from step to step: the list names its elements only)
              products[key] = {op, nz, list, flags & ~had};
            }
          }
          flags |= more;
          MRec& c = append(op);
          c.w[1] = slot(out);
          c.w[2] = x;
          c.w[3] = y;
          c.w[4] = (uint32_t)rows | (uint32_t)cols << 8 | (uint32_t)K << 16 | (uint32_t)nz << 24;
          c.w[5] = (uint32_t)xi | (uint32_t)xq << 16;
          c.w[6] = (uint32_t)yq | (uint32_t)yj << 16;
          c.w[8] = (uint32_t)list;
          c.w[9] = row_of(cols);
          c.w[10] = (uint32_t)gate;
          save(c, sv);
        };
        const int r = d.r, c_ = d.c, k = d.k, w = r * c_, n = d.r;
        switch (d.op) {
          case D_GATHER: {
            // elements of slots, and zeros: a list
            std::vector<int32_t> l;
            for (int e = 0; e < f[2]; e++) {
              const int32_t ref = p.args[(size_t)f[1] + (size_t)e];
              if (ref_kind(ref) == RK_SLOT) { l.push_back(ref_index(ref)); continue; }
              const double v = ref_kind(ref) == RK_CONST ? pool_at(ref_index(ref), 0) : 1.0;
              if (v != 0 || std::signbit(v)) break;
              l.push_back((int32_t)kCNone);
            }
            if ((int)l.size() == f[2] && f[2] <= kMaxDim * kMaxDim) {
              const int list = mx->list(l);
              MRec& c = append(M_SELECT);
              c.w[1] = slot(f[0]);
              c.w[2] = c.w[3] = 0;
              c.w[4] = (uint32_t)r | (uint32_t)c_ << 8 | 1u << 16;
              c.w[8] = (uint32_t)list;
              c.w[9] = row_of(c_);
              save(c, f[3]);
              break;
            }
            MRec& c = append(M_GATHER);
            c.w[1] = slot(f[0]);
            c.w[2] = (uint32_t)f[1];
            c.w[3] = (uint32_t)f[2];
            save(c, f[3]);
            break;
          }
          case D_MADD: case D_MSUB: {
            // z = t + B, B + t or B - t right after t's product: one record for both
            const bool t1 = f[1] == last_product, t2 = f[2] == last_product;
            if (last_product != -1 && t1 != t2 && !(t1 && d.op == D_MSUB) && (int)code.size() == last_product_pc + 1) {
              const int32_t other = t1 ? f[2] : f[1];
              const uint32_t kind = ref_kind(other);
              // (its slots must not be an operand's of the product, which other threads still read)
              auto apart = [&](const std::pair<int32_t, int>& in) {
                return ref_kind(in.first) != RK_SLOT || in.first + in.second <= f[0] || f[0] + w <= in.first;
              };
              if (apart(last_in[0]) && apart(last_in[1]) && (kind == RK_SLOT || kind == RK_CONST || kind == RK_OBS)) {
                const int at = last_product_pc;
                uint32_t v = 0;
                if (kind == RK_SLOT) v = slot(other);
                if (kind == RK_CONST) v = (uint32_t)mx->constants(pool, ref_index(other), w);
                MRec& c = code[(size_t)at];
                c.w[0] |= kMPost | (d.op == D_MSUB ? kMPostNeg : 0) | (kind == RK_CONST ? kMPostConst : 0);
                c.w[11] = slot(f[0]);
                c.w[12] = v;
                c.w[13] = (uint32_t)f[3];
                if (kind == RK_OBS) mx->use(mx->stage(true, ref_index(other), w, at), at, 12);
                break;
              }
            }
            const uint32_t x = operand(f[1], w, 2, kMConstX), y = operand(f[2], w, 3, kMConstY);
            if (d.op == D_MSUB) flags |= kCNeg;
            MRec& c = append((flags & (kMConstX | kMConstY)) ? M_ADDC : M_ADD);
            c.w[1] = slot(f[0]);
            c.w[2] = x;
            c.w[3] = y;
            c.w[4] = (uint32_t)w;
            save(c, f[3]);
            break;
          }
          case D_MSCALE: {
            const uint32_t x = operand(f[1], 1, 2, kMConstX), y = operand(f[2], w, 3, kMConstY);
            MRec& c = append(M_SCALE);
            c.w[1] = slot(f[0]);
            c.w[2] = x;
            c.w[3] = y;
            c.w[4] = (uint32_t)w;
            save(c, f[3]);
            break;
          }
          case D_MATMUL:
            mm(f[0], f[1], r * k, k, 1, f[2], k * c_, c_, 1, r, c_, k, 0, 0, f[3]);
            last_product = f[0];
            last_product_pc = (int)code.size() - 1;
            last_in[0] = {f[1], r * k};
            last_in[1] = {f[2], k * c_};
            break;
          case D_INV: case D_DET: case D_LOGDET: {
            const uint32_t x = operand(f[1], n * n, 2, 0);
            MRec& c = append(d.op == D_INV ? M_INV : d.op == D_DET ? M_DET : M_LOGDET);
            c.w[1] = slot(f[0]);
            c.w[2] = x;
            c.w[3] = slot(f[2]);
            c.w[4] = (uint32_t)n | row_of(n) << 8;
            c.w[5] = d.op == D_INV ? kCNone : slot(f[4]);
            c.w[6] = d.op == D_INV ? kCNone : (uint32_t)f[5];
            save(c, f[3]);
            break;
          }
          case D_TRACE: {
            const uint32_t x = operand(f[1], n * n, 2, kMConstX);
            MRec& c = append(M_TRACE);
            c.w[1] = slot(f[0]);
            c.w[2] = x;
            c.w[4] = (uint32_t)n;
            save(c, f[3]);
            break;
          }
          case B_MADD: case B_MSUB:
            for (int side = 1; side <= 2; side++) {
              if (f[side] == -1) continue;
              const bool first = d.flags & side;
              flags = side == 2 && d.op == B_MSUB ? kCNeg : 0;
              MRec& c = append(first ? M_COPY : M_ADD);
              c.w[1] = slot(f[side]);
              c.w[2] = slot(first ? f[0] : f[side]);
              c.w[3] = slot(f[0]);
              c.w[4] = (uint32_t)w;
            }
            break;
          case B_MSCALE: {
            // (f4, the matrix, only when f1 is a target; f3, the scalar, only when f2 is)
            const uint32_t s = f[2] != -1 ? operand(f[3], 1, 5, kMConstX) : kCNone;
            const uint32_t y = f[1] != -1 ? operand(f[4], w, 6, kMConstY) : kCNone;
            flags |= fa | fb;
            MRec& c = append(M_RSCALE);
            c.w[1] = slot(f[0]);
            c.w[2] = slot(f[1]);
            c.w[3] = slot(f[2]);
            c.w[4] = (uint32_t)w;
            c.w[5] = s;
            c.w[6] = y;
            break;
          }
          case B_MATMUL:
            if (f[1] != -1) mm(f[1], f[0], w, c_, 1, f[4], k * c_, 1, c_, r, k, c_, kMGateX | (fa ? 0 : kMAcc), w, -1);
            if (ok && f[2] != -1) mm(f[2], f[3], r * k, 1, k, f[0], w, c_, 1, k, c_, r, kMGateY | (fb ? 0 : kMAcc), w, -1);
            break;
          case B_INV:
            if (f[1] == -1) break;
            mm(f[2], f[0], n * n, n, 1, f[5], n * n, 1, n, n, n, n, kMGateX, n * n, -1);
            if (ok) mm(f[1], f[5], n * n, 1, n, f[2], n * n, n, 1, n, n, n, kMGateY | kCNeg | (fa ? 0 : kMAcc), n * n, -1);
            break;
          case B_DET: case B_LOGDET: {
            if (f[1] == -1) break;
            const uint32_t z = d.op == B_DET ? operand(f[5], 1, 5, 0) : kCNone, y = operand(f[6], n * n, 6, 0);
            flags |= fa;
            MRec& c = append(M_RDET);
            c.w[1] = slot(f[0]);
            c.w[2] = slot(f[1]);
            c.w[4] = (uint32_t)n | row_of(n) << 8;
            c.w[5] = z;
            c.w[6] = y;
            break;
          }
          case B_TRACE: {
            if (f[1] == -1) break;
            flags |= fa;
            MRec& c = append(M_RTRACE);
            c.w[1] = slot(f[0]);
            c.w[2] = slot(f[1]);
            c.w[4] = (uint32_t)n;
            break;
          }
          case B_GATHER: {
            MRec& c = append(M_RGATHER);
            c.w[1] = slot(f[0]);
            c.w[2] = (uint32_t)f[1];
            c.w[3] = (uint32_t)f[2];
            break;
          }
          case B_SCATTER: {
            if (f[1] == -1) break;
            if (fa) {  // a first contribution by a one-to-one map: each target's element, or 0
              std::vector<int32_t> l((size_t)f[4], (int32_t)kCNone);
              bool once = true;
              for (int e = 0; e < f[2]; e++) {
                int32_t& t = l[(size_t)p.args[(size_t)f[3] + (size_t)e]];
                once = once && t == (int32_t)kCNone;
                t = ref_index(f[0]) + e;
              }
              int tr = f[4], tc = 1;  // (a shape of f[4] elements within the fields' range)
              for (int q = 2; q <= kMaxDim && tr > kMaxDim; q++)
                if (f[4] % q == 0) { tr = f[4] / q; tc = q; }
              if (once && tr <= kMaxDim) {
                const int list = mx->list(l);
                MRec& c = append(M_RSELECT);
                c.w[1] = slot(f[1]);
                c.w[2] = c.w[3] = 0;
                c.w[4] = (uint32_t)tr | (uint32_t)tc << 8 | 1u << 16;
                c.w[8] = (uint32_t)list;
                c.w[9] = row_of(tc);
                break;
              }
            }
            flags |= fa;
            MRec& c = append(M_RSCATTER);
            c.w[1] = slot(f[0]);
            c.w[2] = slot(f[1]);
            c.w[3] = (uint32_t)f[3];
            c.w[4] = (uint32_t)f[2];
            c.w[5] = (uint32_t)f[4];
            break;
          }
          default: return none;
        }
        if (!ok) return none;
        break;
      }
    }
    if (d.op != D_SEED && d.op != D_LOAD) pending_seed = -1;
  }
  if (loop_pc >= 0 || !copies.empty()) return none;
  rec(C_END);
  if (mx) return code;
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
  std::vector<MRec> kept;
  for (size_t q = 0; q < code.size(); q++) {
    newpc[q] = (uint32_t)kept.size();
    if (!dead[q]) kept.push_back(code[q]);
  }
  for (MRec& c : kept)
    if ((c.w[0] & 0xff) == C_LOOP) c.w[4] = newpc[c.w[4]];
  return kept;
}

// The slot that a record writes, when it writes one value or none (kCNone); all = false when it may
// write others.
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
    bool all;
    const uint32_t s = writes(c, &all);
    if (s != kCNone) write(s, pc);
    if (all || op == C_LOOP || op == C_ENDLOOP) continue;
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
    if ((code[(size_t)u.writer].w[0] & 0xff) == C_FETCH) continue;  // its copy lands later
    if ((int)rcp.size() >= kCMaxReciprocals) break;
    make[u.writer] = c.w[3];
    rcp[c.w[3]] = (uint32_t)(*n_slots)++ * kCSlotUnit;
  }
  if (rcp.empty()) return;
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

// What the records add to the plan's work (less than 0).  The planner counts a lane-level division as
// the IEEE division and a body's with a reciprocal of its own, kept for the reverse rule; here every
// division is by a reciprocal, shared or its own.  And it counts every term of a product or of a
// scaling's adjoint; here the terms of a constant's zeros are left out, and a selection has none.
template <typename R>
void recount(Plan& p, const std::vector<R>& code, const Matrices* mx) {
  const double whole = cost::kRcpNewton + cost::kDivStep;
  double points = 1;
  bool loop = false;
  p.records_fwd = p.records_rev = 0;
  for (const R& c : code) {
    const uint32_t* w = c.w;
    const uint32_t op = w[0] & 0xff;
    if (op == C_LOOP) { loop = true; points = (double)w[1]; }
    if (op == C_ENDLOOP) { loop = false; points = 1; }
    if (op == C_RCP) p.records_fwd += points * cost::kRcpNewton;
    if (op == C_DIV) p.records_fwd += points * ((w[4] != kCNone ? cost::kDivStep : whole) - (loop ? whole : cost::kDiv));
    if (op == R_DIV) p.records_rev += points * ((w[7] != kCNone ? cost::kDivStep : whole) - (loop ? cost::kDivStep : cost::kDiv));
    if (op >= M_FSPARSE && op <= M_RSELECT && (w[0] & (kMConstX | kMConstY))) {
      const uint32_t e = (w[4] & 0xff) * ((w[4] >> 8) & 0xff), K = (w[4] >> 16) & 0xff;
      double terms = 0;
      for (uint32_t q = 0; op <= M_RSPARSE && q < e * (w[4] >> 24); q++) {
        const uint32_t x = (uint32_t)mx->lists[w[8] + q];
        terms += x != kCNone && x != kMSplit;
      }
      (op == M_FSPARSE || op == M_SELECT ? p.records_fwd : p.records_rev) += terms - (double)e * K;
    }
    if (op == M_RSCALE && w[2] != kCNone && (w[0] & kMConstY))
      for (uint32_t q = 0; q < w[4]; q++) p.records_rev -= mx->consts[w[6] + q] == 0;
  }
}

// Inserts the staged operands' copies and waits, and gives them slots from `slots` on; returns
// the slots in use.
int place_stages(std::vector<MRec>& code, Matrices& mx, int slots) {
  // a copy runs kMAhead records before its first use, after the reverse sweep has begun if its
  // source is the workspace (the forward sweep has then stored it)
  const int rev = mx.rev_begin < 0 ? (int)code.size() : mx.rev_begin;
  for (auto& s : mx.stages) s.fetch_at = std::min(s.use_first, std::max(s.from_obs ? 0 : rev, s.use_first - kMAhead));
  std::vector<int> order(mx.stages.size());
  for (size_t k = 0; k < order.size(); k++) order[k] = (int)k;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return mx.stages[(size_t)a].fetch_at < mx.stages[(size_t)b].fetch_at; });
  std::vector<int> busy_until;  // per staging slot: the last record that reads it
  for (int k : order) {
    Matrices::Stage& s = mx.stages[(size_t)k];
    int run = 0, at = -1;
    for (int q = 0; q < (int)busy_until.size() && at < 0; q++) {
      run = busy_until[(size_t)q] < s.fetch_at ? run + 1 : 0;
      if (run == s.width) at = q - s.width + 1;
    }
    if (at < 0) {
      at = (int)busy_until.size() - run;
      busy_until.resize((size_t)(at + s.width), -1);
    }
    for (int q = at; q < at + s.width; q++) busy_until[(size_t)q] = s.use_last;
    s.slot = slots + at;
    for (const auto& u : s.patches) code[(size_t)u.first].w[u.second] = (uint32_t)s.slot * kCSlotUnit;
  }
  std::vector<MRec> out;
  std::vector<int> commits_at;               // commits so far, after the copy of stage k
  commits_at.assign(mx.stages.size(), 0);
  std::multimap<int, int> need;              // record -> stage first read there
  for (size_t k = 0; k < mx.stages.size(); k++) need.insert({mx.stages[k].use_first, (int)k});
  size_t next = 0;
  int commits = 0;
  for (int pc = 0; pc < (int)code.size(); pc++) {
    while (next < order.size() && mx.stages[(size_t)order[next]].fetch_at == pc) {
      const Matrices::Stage& s = mx.stages[(size_t)order[next]];
      MRec f;
      f.w[0] = M_FETCH | (s.from_obs ? kMFromObs : 0);
      f.w[1] = (uint32_t)s.slot * kCSlotUnit;
      f.w[2] = (uint32_t)s.src;
      f.w[3] = (uint32_t)s.width;
      out.push_back(f);
      commits_at[(size_t)order[next]] = ++commits;
      next++;
    }
    // the record before the first one that reads a copy waits for it
    const auto range = need.equal_range(pc);
    for (auto it = range.first; it != range.second; ++it) {
      const uint32_t pending = (uint32_t)std::min(commits - commits_at[(size_t)it->second], 7);
      uint32_t& w = out.back().w[0];  // (a copy precedes its use, so there is a record)
      const uint32_t had = (w >> kMWaitShift) & 7u, want = std::min(1 + pending, 7u);
      if (had == 0 || want < had) w = (w & ~(7u << kMWaitShift)) | want << kMWaitShift;
    }
    out.push_back(code[(size_t)pc]);
    if ((code[(size_t)pc].w[0] & 0xff) == C_FETCH && (code[(size_t)pc].w[0] & kCCommit)) commits++;
  }
  code.swap(out);
  return slots + (int)busy_until.size();
}

// A long stream's chunks: the last record of each says so.
template <typename R, size_t CHUNK>
void mark_chunks(std::vector<R>& code) {
  std::vector<R> out;
  R mark;
  mark.w[0] = C_CHUNK;
  for (const R& c : code) {
    if (out.size() % CHUNK == CHUNK - 1) out.push_back(mark);
    out.push_back(c);
  }
  code.swap(out);
}

}  // namespace

void compact_plan(Plan& p, const std::vector<double>& consts) {
  for (Plan& d : p.derive) compact_plan(d, consts);
  p.compact.clear();
  p.matrix.clear();
  p.compact_slots = p.n_slots + kCExtraSlots;
  p.compact_points = 0;
  if (!compact_enabled()) return;
  if (p.has_matrix) {
    // (where a lane's slots leave no room for the constants, the general kernel runs)
    if (p.has_regions || (size_t)p.n_slots * sizeof(double) > (size_t)150 * 1024) return;
    Matrices mx;
    int64_t points = 0;
    std::vector<MRec> code = translate(p, consts, &points, &mx);
    if (code.empty() || mx.consts.size() > kMMaxConsts) return;
    p.matrix_width = 0;
    for (const MRec& c : code)
      if ((c.w[0] & 0xff) >= M_F && (c.w[0] & 0xff) <= M_RSELECT)
        p.matrix_width = std::max(p.matrix_width, (int32_t)((c.w[4] & 0xff) * ((c.w[4] >> 8) & 0xff)));
    recount(p, code, &mx);
    p.matrix_slots = place_stages(code, mx, p.n_slots + kCExtraSlots + mx.temps);
    mark_chunks<MRec, kMChunk>(code);
    for (const MRec& c : code) p.matrix.insert(p.matrix.end(), c.w, c.w + kMatrixWords);
    p.matrix_consts = mx.consts;
    p.matrix_lists = mx.lists;
    return;
  }
  std::vector<CRec> code;
  for (const MRec& m : translate(p, consts, &p.compact_points, nullptr)) {
    CRec c;
    std::copy(m.w, m.w + kCompactWords, c.w);
    code.push_back(c);
  }
  if (code.empty()) return;
  share_reciprocals(code, &p.compact_slots);
  // (a loop is not read in chunks, nor is one of no points, which still has its records)
  const bool loop = std::any_of(code.begin(), code.end(), [](const CRec& c) { return (c.w[0] & 0xff) == C_LOOP; });
  if (loop && code.size() > kCResident) return;
  recount(p, code, nullptr);
  if (code.size() > kCResident) mark_chunks<CRec, kCChunk>(code);
  for (const CRec& c : code) p.compact.insert(p.compact.end(), c.w, c.w + kCompactWords);
}

}  // namespace ndvm
