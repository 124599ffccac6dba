// Test infrastructure: a CPU executor of the compact and matrix records (compact.h), one lane at a
// time and one thread per lane, with K points per pass in a data-axis loop.  Every record is checked
// first: its kind, its slots, workspace elements, constants and list entries, and that no stream
// with a loop is cut into chunks.  Asynchronous copies land when the stream waits for them and the
// slots they write hold NaN until then, so a wait that is missing shows in the results.
//
// Input on stdin:  frontend B P n_obs stream(0 gradient plan, 1 value plan) K / B*P params /
//                  n_obs obs / the program text up to end of input.
// With the argument "apart", a record that does nothing stands between each seed and its loop.
// Output: the kind of the stream (compact, matrix or none) and the entries of its lists, then one line
// per lane: the loss and the P gradient components as C hex floats.  Exit status 5: a record failed a check.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <iostream>
#include <limits>
#include <sstream>
#include <string>
#include <vector>

#include "compact.h"
#include "tape.h"

using namespace ndvm;

namespace {

bool is_zero(double x) { return x == 0.0; }
bool gt_eps(double x) { return x > 1e-8; }
double powi(double a, int n) {
  double z = n == 0 ? 1.0 : a;
  for (int i = 1; i < n; i++) z = z * a;
  return z;
}

struct Bad {
  std::string why;
};

// determinant and inverse by Gauss-Jordan elimination with partial pivoting
double det_inv(std::vector<double> w, int n, std::vector<double>* inv) {
  std::vector<double> v((size_t)(n * n), 0.0);
  for (int i = 0; i < n; i++) v[(size_t)(i * n + i)] = 1.0;
  double d = 1.0;
  for (int c = 0; c < n; c++) {
    int p = c;
    for (int i = c + 1; i < n; i++)
      if (std::fabs(w[(size_t)(i * n + c)]) > std::fabs(w[(size_t)(p * n + c)])) p = i;
    if (p != c) {
      d = -d;
      for (int j = 0; j < n; j++) {
        std::swap(w[(size_t)(p * n + j)], w[(size_t)(c * n + j)]);
        std::swap(v[(size_t)(p * n + j)], v[(size_t)(c * n + j)]);
      }
    }
    const double pv = w[(size_t)(c * n + c)];
    d = d * pv;
    for (int j = 0; j < n; j++) { w[(size_t)(c * n + j)] /= pv; v[(size_t)(c * n + j)] /= pv; }
    for (int i = 0; i < n; i++) {
      const double f = w[(size_t)(i * n + c)];
      if (i == c || f == 0.0) continue;
      for (int j = 0; j < n; j++) {
        w[(size_t)(i * n + j)] -= f * w[(size_t)(c * n + j)];
        v[(size_t)(i * n + j)] -= f * v[(size_t)(c * n + j)];
      }
    }
  }
  if (inv) *inv = v;
  return d;
}

struct Run {
  const Plan& p;
  const bool mx;            // matrix records
  const int K;              // values of a slot
  const int n_slots;
  const std::vector<double>& consts;   // the plan's constant pool
  const std::vector<double>& mconsts;  // the matrix records' constants
  const double* obs;
  const double* ext;        // the regions' blocks, by extended index
  const double* params;
  double* save;
  int64_t save_ld, col;
  double* loss = nullptr;
  double* grad = nullptr;
  std::vector<double> s;
  const double* point[4] = {nullptr, nullptr, nullptr, nullptr};
  bool met = false;         // an infinity or a NaN has been stored in a matrix
  struct Copy { size_t slot; double v; };
  std::vector<std::vector<Copy>> groups;  // committed, not landed
  std::vector<Copy> open;

  Run(const Plan& q, const std::vector<double>& k, const double* o, const double* e, const double* pa, double* sv,
      int64_t ld, int64_t c, int points)
      : p(q), mx(!q.matrix.empty()), K(points), n_slots(mx ? q.matrix_slots : q.compact_slots), consts(k),
        mconsts(q.matrix_consts), obs(o), ext(e), params(pa), save(sv), save_ld(ld), col(c),
        s((size_t)n_slots * (size_t)points, std::numeric_limits<double>::quiet_NaN()) {}

  size_t at(uint32_t w) const { return (size_t)(w / kCSlotUnit) * (size_t)K; }
  double* v(uint32_t w) { return &s[at(w)]; }
  double ld(uint32_t w) const { return s[at(w)]; }
  void st(uint32_t w, double x) {  // outside a loop: every point's copy
    for (int j = 0; j < K; j++) s[at(w) + (size_t)j] = x;
  }
  double& el(uint32_t w, int e) { return s[(size_t)(w / kCSlotUnit) + (size_t)e]; }
  double& saved(uint32_t idx) { return save[(int64_t)idx * save_ld + col]; }
  void see(double x) { met = met || !std::isfinite(x); }
  void land(size_t keep) {
    while (groups.size() > keep) {
      for (const Copy& c : groups.front()) s[c.slot] = c.v;
      groups.erase(groups.begin());
    }
  }
  void copy(uint32_t dst, size_t e, double x) {
    const size_t q = at(dst) + e * (size_t)K;
    s[q] = std::numeric_limits<double>::quiet_NaN();
    open.push_back({q, x});
  }
  void commit() {
    groups.push_back(open);
    open.clear();
  }

  // a scalar record on n values (1 outside a loop); false: not one
  bool scalar(const uint32_t* w, int n) {
    const uint32_t f = w[0], op = f & 0xff;
    double z[4], a[4];
    auto put = [&](uint32_t dst, const double* x) {
      for (int j = 0; j < K; j++) s[at(dst) + (size_t)j] = x[n == K ? j : 0];
    };
    auto update = [&](uint32_t dst, const double* x, const bool* on, bool first) {
      double q[4];
      for (int j = 0; j < n; j++) q[j] = first ? (on[j] ? x[j] : 0.0) : on[j] ? v(dst)[j] + x[j] : v(dst)[j];
      put(dst, q);
    };
    bool on[4];
    for (int j = 0; j < n && op >= R_DIV && op <= R_DSUM; j++) on[j] = !is_zero(v(w[1])[j]);
    auto each = [&](auto&& g) {
      for (int j = 0; j < n; j++) z[j] = g(j);
    };
    switch (op) {
      case C_ARITH:
        each([&](int j) {
          const double x = v(w[2])[j], y = (f & kCHasB) ? v(w[3])[j] : 1.0, c = (f & kCHasC) ? v(w[4])[j] : -0.0;
          return std::fma((f & kCNeg) ? -x : x, (f & kCGate) && is_zero(x) ? 0.0 : y, c);
        });
        break;
      case C_DIV:
        each([&](int j) { return v(w[2])[j] / v(w[3])[j]; });
        if (w[4] == kCNone && w[5] != kCNone) {
          for (int j = 0; j < n; j++) a[j] = 1.0 / v(w[3])[j];
          put(w[5], a);
        }
        if (w[4] != kCNone)
          for (int j = 0; j < n; j++)
            if (v(w[4])[j] != 1.0 / v(w[3])[j] && !std::isnan(v(w[3])[j])) throw Bad{"a shared reciprocal is not the divisor's"};
        break;
      case C_RCP: each([&](int j) { return 1.0 / v(w[2])[j]; }); break;
      case C_POW: each([&](int j) { return std::pow(v(w[2])[j], v(w[3])[j]); }); break;
      case C_EXP: each([&](int j) { return std::exp(v(w[2])[j]); }); break;
      case C_LOG: each([&](int j) { return std::log(gt_eps(v(w[2])[j]) ? v(w[2])[j] : 1e-8); }); break;
      case C_TANH: each([&](int j) { return std::tanh(v(w[2])[j]); }); break;
      case C_SQRT: each([&](int j) { return std::sqrt(gt_eps(v(w[2])[j]) ? v(w[2])[j] : 1e-8); }); break;
      case C_ABS: each([&](int j) { return std::fabs(v(w[2])[j]); }); break;
      case C_POWI: each([&](int j) { return powi(v(w[2])[j], (int)w[6]); }); break;
      case C_SIN: case C_COS:
        for (int j = 0; j < n; j++) a[j] = op == C_SIN ? std::cos(v(w[2])[j]) : std::sin(v(w[2])[j]);
        each([&](int j) { return op == C_SIN ? std::sin(v(w[2])[j]) : std::cos(v(w[2])[j]); });
        if (w[5] != kCNone) put(w[5], a);
        if ((int)w[6] >= 0) saved(w[6]) = a[0];
        break;
      case C_CMP:
        each([&](int j) {
          const double x = v(w[2])[j], y = v(w[3])[j];
          const uint32_t k = (f >> kCCountShift) & 7;
          return (k == 0 ? x < y : k == 1 ? x <= y : k == 2 ? x > y : k == 3 ? x >= y : x == y) ? 1.0 : 0.0;
        });
        break;
      case C_SELECT: each([&](int j) { return !is_zero(v(w[2])[j]) ? v(w[3])[j] : v(w[4])[j]; }); break;
      case R_DIV: {
        double q[4];
        for (int j = 0; j < n; j++) q[j] = v(w[1])[j] / v(w[5])[j];
        if (w[2] != kCNone) update(w[2], q, on, f & kCFirstA);
        if (w[3] != kCNone) {
          for (int j = 0; j < n; j++) z[j] = -(q[j] * v(w[6])[j]);
          update(w[3], z, on, f & kCFirstB);
        }
        return true;
      }
      case R_POW:
        if (w[2] != kCNone) {
          each([&](int j) { return v(w[1])[j] * v(w[5])[j] * v(w[6])[j] / v(w[4])[j]; });
          update(w[2], z, on, f & kCFirstA);
        }
        if (w[3] != kCNone) {
          each([&](int j) { return v(w[1])[j] * v(w[6])[j] * std::log(v(w[4])[j]); });
          update(w[3], z, on, f & kCFirstB);
        }
        return true;
      case R_TANH: each([&](int j) { return v(w[1])[j] * (1.0 - v(w[6])[j] * v(w[6])[j]); }); update(w[2], z, on, f & kCFirstA); return true;
      case R_LOG: each([&](int j) { return gt_eps(v(w[4])[j]) ? v(w[1])[j] / v(w[4])[j] : 0.0; }); update(w[2], z, on, f & kCFirstA); return true;
      case R_ABS:
        each([&](int j) { const double g = v(w[1])[j], x = v(w[4])[j]; return x > 0 ? g : x < 0 ? -g : g * 0.0; });
        update(w[2], z, on, f & kCFirstA);
        return true;
      case R_SQRT:
        each([&](int j) { return gt_eps(v(w[4])[j]) ? v(w[1])[j] / (2.0 * v(w[6])[j]) : 0.0; });
        update(w[2], z, on, f & kCFirstA);
        return true;
      case R_POWI: {
        const int k = (int)w[7];
        each([&](int j) { return k > 0 ? v(w[1])[j] * ((double)k * powi(v(w[4])[j], k - 1)) : 0.0; });
        update(w[2], z, on, f & kCFirstA);
        return true;
      }
      case R_SELECT: {
        bool ta[4], tb[4];
        for (int j = 0; j < n; j++) {
          const bool taken = !is_zero(v(w[4])[j]);
          z[j] = v(w[1])[j];
          ta[j] = on[j] && taken;
          tb[j] = on[j] && !taken;
        }
        if (w[2] != kCNone) update(w[2], z, ta, f & kCFirstA);
        if (w[3] != kCNone) update(w[3], z, tb, f & kCFirstB);
        return true;
      }
      case R_DSUM: each([&](int j) { return v(w[1])[j] * v(w[4])[j]; }); update(w[2], z, on, f & kCFirstA); return true;
      default: return false;
    }
    put(w[1], z);
    if (f & kCSave) saved(w[7]) = z[0];
    return true;
  }

  void outer(const uint32_t* w) {
    switch (w[0] & 0xff) {
      case C_FETCH:
        for (uint32_t e = 0; e < ((w[0] >> kCCountShift) & 7); e++) copy(w[1 + 2 * e], 0, saved(w[2 + 2 * e]));
        if (w[0] & kCCommit) commit();
        if (w[0] & kCWait) land((w[0] >> kCPendingShift) & 7);
        break;
      case C_OBS:
        for (uint32_t e = 0; e < ((w[0] >> kCCountShift) & 7); e++)
          for (int j = 0; j < K; j++) v(w[1 + 2 * e])[j] = point[j][w[2 + 2 * e]];
        break;
      case C_LOADC: {
        const uint64_t b = (uint64_t)w[2] | (uint64_t)w[3] << 32;
        double x;
        std::memcpy(&x, &b, 8);
        st(w[1], x);
        break;
      }
      case C_LOADP: st(w[1], params[w[2]]); break;
      case C_LOADO: st(w[1], obs[w[2]]); break;
      case C_LOADS: st(w[1], saved(w[2])); break;
      case C_ZERO: for (uint32_t e = 0; e < w[2]; e++) st(w[1] + e * kCSlotUnit, 0.0); break;
      case C_SEED: st(w[1], 1.0); break;
      case C_GREDUCE:
        for (uint32_t e = 0; e < w[2]; e++) {
          double t = v(w[1] + e * kCSlotUnit)[0];
          for (int j = 1; j < K; j++) t = t + v(w[1] + e * kCSlotUnit)[j];
          st(w[1] + e * kCSlotUnit, t);
        }
        break;
      case C_LOSS: if (loss) *loss = ld(w[1]); break;
      case C_GRAD: if (grad) grad[w[2]] = w[1] == kCNone ? 0.0 : ld(w[1]); break;
      default: throw Bad{"unknown record " + std::to_string(w[0] & 0xff)};
    }
  }

  double operand(uint32_t w, bool c, int e) { return c ? mconsts[(size_t)w + (size_t)e] : el(w, e); }
  bool all_zero(uint32_t w, int n) {
    for (int e = 0; e < n; e++)
      if (!is_zero(el(w, e))) return false;
    return true;
  }

  void product(const uint32_t* w) {
    const uint32_t f = w[0], op = f & 0xff;
    const bool rev = (op >= M_R && op <= M_R8) || op == M_RSPARSE || op == M_RSELECT;
    const bool list = op == M_FSPARSE || op == M_RSPARSE, select = op == M_SELECT || op == M_RSELECT;
    const bool cx = f & kMConstX, cy = f & kMConstY;
    const int rows = w[4] & 0xff, cols = (w[4] >> 8) & 0xff, k = (w[4] >> 16) & 0xff, nz = (int)(w[4] >> 24);
    const int xi = w[5] & 0xffff, xq = (int)(w[5] >> 16), yq = w[6] & 0xffff, yj = (int)(w[6] >> 16);
    const bool all = met && (cx || cy);
    const int32_t* l = p.matrix_lists.data() + w[8];
    std::vector<double> zs((size_t)(rows * cols));
    for (int e = 0; e < rows * cols; e++) {
      const int i = e / cols, j = e - i * cols;
      const double s0 = rev && (f & kMAcc) ? ((f & kCNeg) ? -el(w[1], e) : el(w[1], e)) : -0.0;
      double z = s0;
      if (select && !all) {
        const uint32_t q = (uint32_t)l[e];
        z = q == kCNone ? 0.0 : el((f & kMOtherY) ? w[3] : w[2], (int)q);
      } else if (list && !all) {
        double odd = -0.0;
        bool second = false;
        for (int u = 0; u < nz; u++) {
          const uint32_t q = (uint32_t)l[e * nz + u];
          if (q == kCNone) break;
          if (q == kMSplit) { second = true; continue; }
          const double c = mconsts[q & 0xffff];
          const double o = operand((f & kMOtherY) ? w[3] : w[2], cx && cy, (int)(q >> 16));
          if (second) odd = std::fma(c, o, odd);
          else z = std::fma(c, o, z);
        }
        if (f & kMChains) z = z + odd;
        if (!(f & kMAcc) && is_zero(z)) z = 0.0;
      } else {
        double odd = -0.0;
        for (int q = 0; q < k; q++) {
          const double x = operand(w[2], cx, i * xi + q * xq), y = operand(w[3], cy, q * yq + j * yj);
          if (k > 8 && q % 2 == 1) odd = std::fma(x, y, odd);
          else z = std::fma(x, y, z);
        }
        if (k > 8) z = z + odd;
      }
      if (rev && std::isnan(z) && (f & (kMGateX | kMGateY)) && all_zero((f & kMGateX) ? w[2] : w[3], (int)w[10]))
        z = (f & kMAcc) ? s0 : 0.0;
      see(z);
      zs[(size_t)e] = rev && (f & kCNeg) ? -z : z;
      if (rev) el(w[1], e) = zs[(size_t)e];  // (the device's order: an element is stored before the next is computed)
    }
    if (rev) return;
    for (int e = 0; e < rows * cols; e++) {
      el(w[1], e) = zs[(size_t)e];
      if (f & kCSave) saved(w[7] + (uint32_t)e) = zs[(size_t)e];
      if (f & kMPost) {
        const double c = operand(w[12], f & kMPostConst, e);
        const double y = (f & kMPostNeg) ? c - zs[(size_t)e] : c + zs[(size_t)e];
        see(y);
        el(w[11], e) = y;
        if ((int)w[13] >= 0) saved(w[13] + (uint32_t)e) = y;
      }
    }
  }

  void matrix(const uint32_t* w) {
    const uint32_t f = w[0], op = f & 0xff;
    const bool fa = f & kCFirstA, fb = f & kCFirstB;
    const int n = (int)w[4], d = (int)(w[4] & 0xff);
    auto put = [&](uint32_t dst, int e, double x) {
      see(x);
      el(dst, e) = x;
      if (f & kCSave) saved(w[7] + (uint32_t)e) = x;
    };
    auto element = [&](int32_t ref) {
      const int32_t i = ref_index(ref);
      switch (ref_kind(ref)) {
        case RK_SLOT: return s[(size_t)i];
        case RK_CONST: return consts[(size_t)i];
        case RK_OBS: return obs[i];
        case RK_SAVE: return saved((uint32_t)i);
        default: return params[i];
      }
    };
    auto run_of = [&](uint32_t src) {
      std::vector<double> m((size_t)(d * d));
      for (int e = 0; e < d * d; e++) m[(size_t)e] = el(src, e);
      return m;
    };
    if (op >= M_F && op <= M_RSELECT) return product(w);
    switch (op) {
      case M_ADD: case M_ADDC: case M_COPY:
        for (int e = 0; e < n; e++) {
          const double x = operand(w[2], f & kMConstX, e), y = op == M_COPY ? x : operand(w[3], f & kMConstY, e);
          put(w[1], e, op == M_COPY ? ((f & kCNeg) ? -x : x) : (f & kCNeg) ? x - y : x + y);
        }
        break;
      case M_SCALE: {
        const double c = operand(w[2], f & kMConstX, 0);
        for (int e = 0; e < n; e++) put(w[1], e, c * operand(w[3], f & kMConstY, e));
        break;
      }
      case M_INV: case M_DET: case M_LOGDET: {
        std::vector<double> inv;
        const double t = det_inv(run_of(w[2]), d, &inv);
        if (op != M_INV) {
          el(w[1], 0) = op == M_DET ? t : std::log(t);
          if (f & kCSave) saved(w[7]) = el(w[1], 0);
        }
        for (int e = 0; e < d * d; e++) {
          if (op == M_INV) { put(w[1], e, inv[(size_t)e]); continue; }
          if (w[5] != kCNone) { see(inv[(size_t)e]); el(w[5], e) = inv[(size_t)e]; }
          if ((int)w[6] >= 0) saved(w[6] + (uint32_t)e) = inv[(size_t)e];
        }
        break;
      }
      case M_TRACE: {
        double t = operand(w[2], f & kMConstX, 0);
        for (int i = 1; i < n; i++) t = t + operand(w[2], f & kMConstX, i * n + i);
        el(w[1], 0) = t;
        if (f & kCSave) saved(w[7]) = t;
        break;
      }
      case M_GATHER:
        for (uint32_t e = 0; e < w[3]; e++) put(w[1], (int)e, element(p.args[w[2] + e]));
        break;
      case M_FETCH:
        for (uint32_t e = 0; e < w[3]; e++) copy(w[1], e, (f & kMFromObs) ? obs[w[2] + e] : saved(w[2] + e));
        commit();
        break;
      case M_RSCALE: {
        const bool zero = all_zero(w[1], n);
        if (w[2] != kCNone) {
          double t = fa ? -0.0 : ld(w[2]);
          if (zero) { if (fa) t = 0.0; }
          else
            for (int e = 0; e < n; e++) {
              const double x = operand(w[6], f & kMConstY, e);
              if (met || !(f & kMConstY) || !is_zero(x)) t = std::fma(el(w[1], e), x, t);
            }
          el(w[2], 0) = t;
        }
        if (w[3] != kCNone)
          for (int e = 0; e < n; e++) {
            if (zero) { if (fb) el(w[3], e) = 0.0; continue; }
            el(w[3], e) = std::fma(operand(w[5], f & kMConstX, 0), el(w[1], e), fb ? -0.0 : el(w[3], e));
            see(el(w[3], e));
          }
        break;
      }
      case M_RDET: {
        const double g = ld(w[1]), fac = w[5] != kCNone ? g * ld(w[5]) : g;
        for (int e = 0; e < d * d; e++) {
          if (is_zero(g)) { if (fa) el(w[2], e) = 0.0; continue; }
          el(w[2], e) = std::fma(fac, el(w[6], (e % d) * d + e / d), fa ? -0.0 : el(w[2], e));
          see(el(w[2], e));
        }
        break;
      }
      case M_RTRACE:
        if (fa) for (int e = 0; e < n * n; e++) el(w[2], e) = 0.0;
        if (!is_zero(ld(w[1])))
          for (int i = 0; i < n; i++) { el(w[2], i * n + i) += ld(w[1]); see(el(w[2], i * n + i)); }
        break;
      case M_RGATHER: {
        const bool zero = all_zero(w[1], (int)w[3]);
        for (uint32_t e = 0; e < w[3]; e++) {
          const int32_t t = p.args[w[2] + 2 * e];
          if (t == -1) continue;
          double& q = s[(size_t)ref_index(t)];
          const bool first = p.args[w[2] + 2 * e + 1] != 0;
          if (zero) { if (first) q = 0.0; }
          else q = first ? el(w[1], (int)e) : q + el(w[1], (int)e);
        }
        break;
      }
      case M_RSCATTER:
        if (fa) for (uint32_t e = 0; e < w[5]; e++) el(w[2], (int)e) = 0.0;
        for (uint32_t e = 0; e < w[4]; e++) {
          double& q = el(w[2], p.args[w[3] + e]);
          q = q + el(w[1], (int)e);
          see(q);
        }
        break;
      default:
        if (op == C_FETCH || op >= C_END || !scalar(w, 1)) outer(w);
    }
    const uint32_t wait = (f >> kMWaitShift) & 7u;
    if (wait) land(wait == 1 ? 0 : 1);  // (as the kernel: none or one group pending)
  }

  void exec() {
    const uint32_t* code = mx ? p.matrix.data() : p.compact.data();
    const int words = mx ? kMatrixWords : kCompactWords;
    const int n = (int)((mx ? p.matrix.size() : p.compact.size()) / (size_t)words);
    int loop = -1;
    int64_t p0 = 0;
    auto pass = [&](const uint32_t* w) {  // the points from p0 on
      for (int j = 0; j < K; j++) {
        const int64_t q = p0 + j, N = w[1];
        s[at(w[5]) + (size_t)j] = q < N ? 1.0 : 0.0;
        point[j] = ((w[0] & kCExt) ? ext : obs) + ((int64_t)w[3] + (q < N ? q : N - 1) * (int64_t)w[2]);
      }
    };
    for (int pc = 0; pc < n; pc++) {
      const uint32_t* w = code + (size_t)pc * (size_t)words;
      const uint32_t op = w[0] & 0xff;
      if (op == C_END) return;
      if (op == C_CHUNK) { commit(); land(0); continue; }
      if (mx) {
        const bool product_record = op >= M_F && op <= M_RSELECT;
        matrix(w);
        const uint32_t wait = (w[0] >> kMWaitShift) & 7u;
        if (product_record && wait) land(wait == 1 ? 0 : 1);
        continue;
      }
      if (op == C_LOOP) {
        if (w[1] == 0) { pc = (int)w[4]; continue; }
        loop = pc;
        p0 = 0;
        pass(w);
      } else if (op == C_ENDLOOP) {
        const uint32_t* l = code + (size_t)loop * (size_t)words;
        p0 += K;
        if (p0 < (int64_t)l[1]) { pass(l); pc = loop; }
        else loop = -1;
      } else if (!scalar(w, loop >= 0 ? K : 1)) {
        outer(w);
      }
    }
    throw Bad{"no end record"};
  }
};

// The checks of a stream's records.
void check(const Plan& p, size_t n_consts) {
  for (const Plan& d : p.derive) check(d, n_consts);
  auto need = [](bool ok, const char* what, size_t pc) {
    if (!ok) throw Bad{std::string(what) + " at record " + std::to_string(pc)};
  };
  const bool mx = !p.matrix.empty();
  const std::vector<uint32_t>& code = mx ? p.matrix : p.compact;
  const size_t words = mx ? kMatrixWords : kCompactWords, n = code.size() / words;
  const uint32_t slots = (uint32_t)(mx ? p.matrix_slots : p.compact_slots);
  bool loops = false, chunks = false, open = false;
  for (size_t pc = 0; pc < n; pc++) {
    const uint32_t* w = &code[pc * words];
    const uint32_t f = w[0], op = f & 0xff;
    auto slot = [&](uint32_t x, uint32_t width, const char* what) {
      need(x % kCSlotUnit == 0 && x / kCSlotUnit + width <= slots, what, pc);
    };
    auto maybe = [&](uint32_t x, uint32_t width, const char* what) { if (x != kCNone) slot(x, width, what); };
    auto save = [&](uint32_t idx, uint32_t width) { need((int64_t)idx + width <= p.n_save, "workspace element", pc); };
    auto matrix = [&](uint32_t x, bool c, uint32_t width, const char* what) {
      if (c) need(x + width <= p.matrix_consts.size(), what, pc);
      else slot(x, width, what);
    };
    need(op < C_NOPS, "record kind", pc);
    loops |= op == C_LOOP;
    chunks |= op == C_CHUNK;
    switch (op) {
      case C_ARITH:
        for (int k = 1; k <= 4; k++) slot(w[k], 1, "slot");
        if (f & kCSave) save(w[7], 1);
        break;
      case C_FETCH: case C_OBS:
        need(((f >> kCCountShift) & 7) <= (uint32_t)kCCopies, "copies", pc);
        for (uint32_t e = 0; e < ((f >> kCCountShift) & 7); e++) {
          slot(w[1 + 2 * e], 1, "copy's slot");
          if (op == C_FETCH) save(w[2 + 2 * e], 1);
        }
        need(op == C_FETCH || open, "observations outside a loop", pc);
        break;
      case C_DIV: case C_RCP: case C_POW: case C_EXP: case C_LOG: case C_TANH: case C_SQRT: case C_ABS: case C_SIN:
      case C_COS: case C_POWI: case C_CMP: case C_SELECT:
        slot(w[1], 1, "result");
        slot(w[2], 1, "operand");
        if (op == C_DIV || op == C_POW || op == C_CMP || op == C_SELECT) slot(w[3], 1, "operand");
        if (op == C_DIV) maybe(w[4], 1, "reciprocal");
        if (op == C_SELECT) slot(w[4], 1, "operand");
        if (op == C_DIV || op == C_SIN || op == C_COS) maybe(w[5], 1, "auxiliary slot");
        if ((op == C_SIN || op == C_COS) && (int)w[6] >= 0) save(w[6], 1);
        if (f & kCSave) save(w[7], 1);
        break;
      case R_DIV: case R_POW: case R_TANH: case R_LOG: case R_ABS: case R_SQRT: case R_POWI: case R_SELECT: case R_DSUM:
        slot(w[1], 1, "adjoint");
        for (int k = 2; k <= (op == R_POWI ? 6 : 7); k++) maybe(w[k], 1, "reverse operand");
        break;
      case C_LOOP:
        need(!open && w[4] < n && (code[w[4] * words] & 0xff) == C_ENDLOOP, "loop", pc);
        slot(w[5], 1, "validity");
        open = true;
        break;
      case C_ENDLOOP: need(open, "loop's end", pc); open = false; break;
      case C_LOADC: case C_LOADP: case C_LOADO: case C_LOADS: case C_SEED: case C_LOSS:
        slot(w[1], 1, "slot");
        if (op == C_LOADP) need(w[2] < (uint32_t)p.n_params, "parameter", pc);
        if (op == C_LOADS) save(w[2], 1);
        break;
      case C_ZERO: case C_GREDUCE: slot(w[1], w[2], "slots"); break;
      case C_GRAD: maybe(w[1], 1, "gradient"); need(w[2] < (uint32_t)p.n_params, "parameter", pc); break;
      case C_CHUNK: case C_END: break;
      case M_ADD: case M_COPY: case M_ADDC:
        slot(w[1], w[4], "result");
        matrix(w[2], f & kMConstX, w[4], "operand");
        matrix(w[3], f & kMConstY, w[4], "operand");
        if (f & kCSave) save(w[7], w[4]);
        break;
      case M_SCALE:
        slot(w[1], w[4], "result");
        matrix(w[2], f & kMConstX, 1, "scalar");
        matrix(w[3], f & kMConstY, w[4], "operand");
        if (f & kCSave) save(w[7], w[4]);
        break;
      case M_INV: case M_DET: case M_LOGDET: {
        const uint32_t d = w[4] & 0xff;
        slot(w[1], op == M_INV ? d * d : 1, "result");
        slot(w[2], d * d, "operand");
        maybe(w[3], 1, "scratch");
        maybe(w[5], d * d, "inverse");
        if (op != M_INV && (int)w[6] >= 0) save(w[6], d * d);
        if (f & kCSave) save(w[7], op == M_INV ? d * d : 1);
        break;
      }
      case M_TRACE:
        slot(w[1], 1, "result");
        matrix(w[2], f & kMConstX, w[4] * w[4], "operand");
        if (f & kCSave) save(w[7], 1);
        break;
      case M_GATHER:
        slot(w[1], w[3], "result");
        need(w[2] + w[3] <= p.args.size(), "list", pc);
        if (f & kCSave) save(w[7], w[3]);
        break;
      case M_FETCH:
        slot(w[1], w[3], "copies");
        if (!(f & kMFromObs)) save(w[2], w[3]);
        break;
      case M_RSCALE:
        slot(w[1], w[4], "adjoint");
        if (w[2] != kCNone) { slot(w[2], 1, "target"); matrix(w[6], f & kMConstY, w[4], "operand"); }
        if (w[3] != kCNone) { slot(w[3], w[4], "target"); matrix(w[5], f & kMConstX, 1, "scalar"); }
        break;
      case M_RDET: {
        const uint32_t d = w[4] & 0xff;
        slot(w[1], 1, "adjoint");
        slot(w[2], d * d, "target");
        maybe(w[5], 1, "determinant");
        slot(w[6], d * d, "inverse");
        break;
      }
      case M_RTRACE: slot(w[1], 1, "adjoint"); slot(w[2], w[4] * w[4], "target"); break;
      case M_RGATHER:
        slot(w[1], w[3], "adjoint");
        need(w[2] + 2 * w[3] <= p.args.size(), "list", pc);
        break;
      case M_RSCATTER:
        slot(w[1], w[4], "adjoint");
        slot(w[2], w[5], "target");
        need(w[3] + w[4] <= p.args.size(), "list", pc);
        break;
      default: {  // products
        need(mx && op >= M_F && op <= M_RSELECT, "record kind", pc);
        const uint32_t rows = w[4] & 0xff, cols = (w[4] >> 8) & 0xff, k = (w[4] >> 16) & 0xff, nz = w[4] >> 24;
        const bool list = op == M_FSPARSE || op == M_RSPARSE, select = op == M_SELECT || op == M_RSELECT;
        const bool cx = f & kMConstX, cy = f & kMConstY;
        const uint32_t wx = (rows - 1) * (w[5] & 0xffff) + (k - 1) * (w[5] >> 16) + 1,
                       wy = (k - 1) * (w[6] & 0xffff) + (cols - 1) * (w[6] >> 16) + 1;
        need(rows >= 1 && cols >= 1 && k >= 1, "shape", pc);
        slot(w[1], rows * cols, "result");
        if (!select || cx || cy) { matrix(w[2], cx, wx, "operand"); matrix(w[3], cy, wy, "operand"); }
        const uint32_t entries = rows * cols * (list ? nz : select ? 1 : 0);
        need(w[8] + entries <= p.matrix_lists.size() || entries == 0, "list", pc);
        for (uint32_t e = 0; e < entries; e++) {
          const uint32_t q = (uint32_t)p.matrix_lists[w[8] + e];
          if (q == kCNone || (list && q == kMSplit)) continue;
          const bool other_y = f & kMOtherY;
          if (list) {
            need((q & 0xffff) < p.matrix_consts.size(), "list's constant", pc);
            matrix(other_y ? w[3] : w[2], cx && cy, (q >> 16) + 1, "list's operand");
          } else {
            slot(other_y ? w[3] : w[2], q + 1, "list's operand");
          }
        }
        if (op >= M_F && op <= M_F8) need((op - M_F == 0 ? k > 8 : op - M_F == k), "terms", pc);
        if (op >= M_R && op <= M_R8) need((op - M_R == 0 ? k > 8 : op - M_R == k), "terms", pc);
        if (f & kCSave) save(w[7], rows * cols);
        if (f & kMPost) {
          slot(w[11], rows * cols, "sum");
          matrix(w[12], f & kMPostConst, rows * cols, "sum's operand");
          if ((int)w[13] >= 0) save(w[13], rows * cols);
        }
      }
    }
  }
  need(!open, "a loop is open", n);
  need(!(loops && chunks), "a stream with a loop is cut into chunks", n);
  need(n == 0 || (code[(n - 1) * words] & 0xff) == C_END, "no end record", n);
}

// an instruction that zeroes no slots ahead of every loop
void part_seeds(Plan& p) {
  std::vector<DInst> out;
  std::vector<int32_t> at;
  for (const DInst& d : p.code) {
    if (d.op == D_LOOP) {
      DInst z;
      z.op = D_ZERO;
      z.f[0] = mkref(RK_SLOT, 0);
      z.f[1] = 0;
      out.push_back(z);
    }
    at.push_back((int32_t)out.size());
    out.push_back(d);
  }
  for (DInst& d : out) {
    if (d.op == D_LOOP) d.f[3] = at[(size_t)d.f[3]];
    if (d.op == D_ENDLOOP) d.f[0] = at[(size_t)d.f[0]];
  }
  p.code.swap(out);
}

}  // namespace

int main(int argc, char** argv) {
  int fe = 0, stream = 0, K = 1;
  int64_t B = 0, P = 0, n_obs = 0;
  std::cin >> fe >> B >> P >> n_obs >> stream >> K;
  std::vector<double> params((size_t)(B * P)), obs((size_t)n_obs);
  std::string word;
  for (auto& v : params) { std::cin >> word; v = std::strtod(word.c_str(), nullptr); }
  for (auto& v : obs) { std::cin >> word; v = std::strtod(word.c_str(), nullptr); }
  std::stringstream rest;
  rest << std::cin.rdbuf();
  const std::string text = rest.str();
  try {
    Builder b;
    std::string err;
    if (fe == 0) trace_scheme(text.data(), text.size(), b, err);
    else trace_bytecode(text.data(), text.size(), b, err);
    if (b.t.loss < 0) { std::fprintf(stderr, "no result: %s\n", err.c_str()); return 2; }
    Plan p = make_plan(b.t, stream == 0);
    if (argc > 1 && std::string(argv[1]) == "apart") part_seeds(p);
    compact_plan(p, b.t.consts);
    check(p, b.t.consts.size() + p.extra_consts.size());
    std::printf("%s %zu\n", !p.matrix.empty() ? "matrix" : !p.compact.empty() ? "compact" : "none", p.matrix_lists.size());
    if (p.matrix.empty() && p.compact.empty()) return 0;
    if (p.n_save > 0 || !p.matrix.empty() || p.compact_points == 0) K = 1;
    std::vector<double> consts = b.t.consts;
    consts.insert(consts.end(), p.extra_consts.begin(), p.extra_consts.end());
    std::vector<double> ext((size_t)(p.n_obs_min + p.derived_elems), 0.0);
    for (size_t k = 0; k < p.derive.size(); k++) {
      const Plan& q = p.derive[k];
      const DeriveInfo& di = p.derive_info[k];
      if (q.compact.empty()) { std::fprintf(stderr, "a derive plan has no records\n"); return 3; }
      for (int64_t pt = 0; pt < di.n_points; pt++)
        Run(q, consts, obs.data(), nullptr, obs.data() + di.base + pt * di.stride, ext.data() + p.n_obs_min + di.offset, di.n_points, pt, 1).exec();
    }
    std::vector<double> ws, g((size_t)P);
    for (int64_t lane = 0; lane < B; lane++) {
      ws.assign((size_t)std::max<int64_t>(p.n_save, 1), std::numeric_limits<double>::quiet_NaN());
      double loss = 0;
      Run r(p, consts, obs.data(), ext.data(), params.data() + lane * P, ws.data(), 1, 0, K);
      r.loss = &loss;
      r.grad = g.data();
      r.exec();
      std::printf("%a", loss);
      for (double v : g) std::printf(" %a", stream == 0 ? v : 0.0);
      std::printf("\n");
    }
  } catch (const Bad& e) {
    std::fprintf(stderr, "record check: %s\n", e.why.c_str());
    return 5;
  } catch (const BuildError& e) {
    std::fprintf(stderr, "build error: %s\n", e.msg.c_str());
    return 2;
  }
  return 0;
}
