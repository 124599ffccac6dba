// Replay of scalar and data-axis tapes: an interpreter of compact records (compact.h).
//
// What bounds these tapes is the interpreter around the arithmetic, not the arithmetic:
// a binary32 operation is one instruction, and a binary64 one holds its scheduler's share
// of the FP64 unit for 64 cycles in which other warps (or points) may issue.  So:
//  - a record is 32 bytes, decoded with one shift-add per operand; the stream sits in
//    shared memory whole (loops) or in double-buffered chunks (long loop-free streams), and
//    the next record is read while the current one runs;
//  - a thread owns a column of slots, 32 threads of a warp adjacent, so an operand is one
//    shared-memory access without bank conflicts;
//  - in a data-axis loop a thread runs K points at once (K = 2 in binary64, 4 in binary32:
//    one 16-byte access per operand), so one record's overhead serves K points and their K
//    independent chains overlap.  Control is uniform over the block: every thread makes the
//    same number of passes, points past the last one repeat it with a zero seed, and a zero
//    adjoint contributes nothing, so only the accumulation of the body's value and of its
//    partials sees the difference.
// Measured on one GB300 against the general kernels (ms): logistic Euler, 16384 lanes x 1000
// steps, 3.05 -> 1.96 in binary64 and 2.01 -> 1.25 in binary32 (102 -> 36 instructions per
// record; one warp per scheduler, so the rest is each record's own latency); an exponential
// fit, 50,001 lanes x 333 points in binary32, 1.33 -> 0.168 (what binds then is issue and the
// shared-memory bandwidth of 16-byte slots); 24 random expressions x 4096 lanes x 256 points in
// binary64 on 8 streams, 2.65 -> 2.30 (the FP64 pipe).  Tried and slower on the logistic tape:
// two records per dispatch, independent or with the second reading the first's result from
// a register (2.23 binary64), and no reading ahead of the next record (2.48).
#include <cuda_runtime.h>

#include <cstdint>

#include "compact.h"
#include "replay.h"
#include "rules.cuh"

namespace ndvm {
namespace {

extern __shared__ __align__(16) unsigned char smem_raw[];

template <typename T, int K>
struct alignas(sizeof(T) * K) Vec {
  T v[K];
};

// log2 of a slot row (32 threads x K values) in units of kCSlotUnit
template <typename T, int K>
__host__ __device__ constexpr int row_shift() {
  return (sizeof(T) * K == 4) ? 0 : (sizeof(T) * K == 8) ? 1 : 2;
}

// Slots and records in shared memory, by 32-bit addresses.  Volatile without a memory clobber:
// the accesses keep their order among themselves, and nothing else touches the slots but the
// asynchronous copies, which are ordered the same way.
__device__ __forceinline__ void ld_shared(unsigned a, double (&x)[1]) { asm volatile("ld.shared.f64 %0, [%1];" : "=d"(x[0]) : "r"(a)); }
__device__ __forceinline__ void ld_shared(unsigned a, double (&x)[2]) {
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(x[0]), "=d"(x[1]) : "r"(a));
}
__device__ __forceinline__ void ld_shared(unsigned a, float (&x)[1]) { asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x[0]) : "r"(a)); }
__device__ __forceinline__ void ld_shared(unsigned a, float (&x)[4]) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]) : "r"(a));
}
__device__ __forceinline__ void st_shared(unsigned a, const double (&x)[1]) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(x[0])); }
__device__ __forceinline__ void st_shared(unsigned a, const double (&x)[2]) {
  asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(x[0]), "d"(x[1]));
}
__device__ __forceinline__ void st_shared(unsigned a, const float (&x)[1]) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(x[0])); }
__device__ __forceinline__ void st_shared(unsigned a, const float (&x)[4]) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]));
}
__device__ __forceinline__ uint4 ld_words(unsigned a) {
  uint4 r;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(a));
  return r;
}

// A thread's slots, and the lane's column of the workspace.
template <typename T, int K>
struct Slots {
  unsigned base;      // shared-memory address of the thread's slot column
  unsigned save_row;  // bytes of a workspace row
  T* save;

  __device__ __forceinline__ unsigned at(uint32_t slot) const { return base + (slot << row_shift<T, K>()); }
  template <int KE>
  __device__ __forceinline__ Vec<T, KE> ld(uint32_t slot) const {
    Vec<T, KE> x;
    ld_shared(at(slot), x.v);
    return x;
  }
  // outside a data-axis loop (KE = 1) every point's copy of the slot gets the value
  template <int KE>
  __device__ __forceinline__ void st(uint32_t slot, const Vec<T, KE>& x) const {
    Vec<T, K> all;
#pragma unroll
    for (int j = 0; j < K; j++) all.v[j] = x.v[KE == K ? j : 0];
    st_shared(at(slot), all.v);
  }
  template <int KE>
  __device__ __forceinline__ void keep(uint32_t flags, uint32_t idx, const Vec<T, KE>& x) const {
    if (K == 1 && (flags & kCSave)) *saved(idx) = x.v[0];  // (a plan that saves runs one point at a time)
  }
  __device__ __forceinline__ T* saved(uint32_t idx) const {
    return reinterpret_cast<T*>(reinterpret_cast<char*>(save) + (uint64_t)idx * save_row);
  }
};

template <typename T, int K>
struct Thread : Slots<T, K> {
  const T* obs;
  const T* params;
  int64_t lane;
  int P, G, grank;
  bool writer;
  const T* point[K];  // observation records of the thread's current points
};

// x + y behind a call: an addition predicated on a flag would take its FP64 slot either way
template <typename T> __device__ __noinline__ T add_call(T x, T y) { return x + y; }

__device__ __forceinline__ double with_sign(double x, uint32_t sign) {  // x, negated when sign's top bit is set
  return __hiloint2double(__double2hiint(x) ^ (int)(sign & 0x80000000u), __double2loint(x));
}
__device__ __forceinline__ float with_sign(float x, uint32_t sign) {
  return __uint_as_float(__float_as_uint(x) ^ (sign & 0x80000000u));
}

// target += v[j] where add[j] (a first contribution stores; where not add[j] it stores 0)
template <typename T, int K, int KE>
__device__ __forceinline__ void update(const Slots<T, K>& t, uint32_t target, const Vec<T, KE>& v, const bool* add, bool first) {
  Vec<T, KE> q;
  if (first) {
#pragma unroll
    for (int j = 0; j < KE; j++) q.v[j] = add[j] ? v.v[j] : (T)0;
  } else {
    q = t.template ld<KE>(target);
#pragma unroll
    for (int j = 0; j < KE; j++)
      if (add[j]) q.v[j] = sizeof(T) == 8 ? add_call(q.v[j], v.v[j]) : q.v[j] + v.v[j];
  }
  t.template st<KE>(target, q);
}
// target += a[j] * b[j] where add[j], in one fused multiply-add
template <typename T, int K, int KE>
__device__ __forceinline__ void update_fma(const Slots<T, K>& t, uint32_t target, const Vec<T, KE>& a, const Vec<T, KE>& b,
                                           const bool* add, bool first) {
  Vec<T, KE> q;
#pragma unroll
  for (int j = 0; j < KE; j++) q.v[j] = neg_zero<T>();
  if (!first) q = t.template ld<KE>(target);
#pragma unroll
  for (int j = 0; j < KE; j++) q.v[j] = fma(add[j] ? a.v[j] : (T)0, add[j] ? b.v[j] : neg_zero<T>(), q.v[j]);
  t.template st<KE>(target, q);
}

// The record kind of the cheap rules (compact.h): no case of a switch.  An absent operand's
// slot is read like any other, which costs less than testing for it, except where a slot
// is four values: there the shared-memory bandwidth binds.
template <typename T, int K, int KE>
__device__ __forceinline__ void arith(const Slots<T, K>& t, const uint4& r0, const uint4& r1) {
  constexpr bool kSkip = KE > 2;
  Vec<T, KE> x = t.template ld<KE>(r0.z), y, c;
  if (kSkip) {
#pragma unroll
    for (int j = 0; j < KE; j++) { y.v[j] = (T)1; c.v[j] = neg_zero<T>(); }
  }
  if (!kSkip || (r0.x & kCHasB)) y = t.template ld<KE>(r0.w);
  if (!kSkip || (r0.x & kCHasC)) c = t.template ld<KE>(r1.x);
  Vec<T, KE> z;
#pragma unroll
  for (int j = 0; j < KE; j++) {
    const T xs = with_sign(x.v[j], r0.x);
    // a zero adjoint leaves c, even against an infinite factor (a zero sum may be +0 for -0)
    const bool off = (r0.x & kCGate) && is_zero(x.v[j]);
    z.v[j] = fma(xs, off ? (T)0 : y.v[j], c.v[j]);
  }
  t.template st<KE>(r0.y, z);
  t.template keep<KE>(r0.x, r1.w, z);
}

#define NDVM_EACH _Pragma("unroll") for (int j = 0; j < KE; j++)

// The functions and the reverse rules that are not in C_ARITH.
template <typename T, int K, int KE>
__device__ __forceinline__ void rule(const Slots<T, K>& t, const uint4& r0, const uint4& r1) {
#define NDVM_FWD1(OPC, EXPR)                       \
  case OPC: {                                      \
    const Vec<T, KE> xv = t.template ld<KE>(r0.z); \
    Vec<T, KE> z;                                  \
    NDVM_EACH { const T x = xv.v[j]; z.v[j] = (EXPR); } \
    t.template st<KE>(r0.y, z);                    \
    t.template keep<KE>(r0.x, r1.w, z);            \
    break;                                         \
  }
  switch (r0.x & 0xff) {
    NDVM_FWD1(C_EXP, fast_exp(x))
    NDVM_FWD1(C_LOG, fast_log(gt_eps(x) ? x : clamp_eps<T>()))
    NDVM_FWD1(C_TANH, tanh(x))
    NDVM_FWD1(C_SQRT, sqrt(gt_eps(x) ? x : clamp_eps<T>()))
    NDVM_FWD1(C_ABS, fabs(x))
    NDVM_FWD1(C_POWI, powi_rep(x, (int)r1.z))
    NDVM_FWD1(C_RCP, div_step_ok((T)1, x) ? rcp_newton(x) : slow_rcp(x))
#undef NDVM_FWD1
    case C_DIV: {
      const Vec<T, KE> x = t.template ld<KE>(r0.z), y = t.template ld<KE>(r0.w);
      Vec<T, KE> z, r;
      if (r1.x != kCNone) {
        r = t.template ld<KE>(r1.x);
        NDVM_EACH z.v[j] = div_by_rcp(x.v[j], y.v[j], r.v[j]);
      } else {
        NDVM_EACH z.v[j] = div_rcp(x.v[j], y.v[j], &r.v[j]);
        if (r1.y != kCNone) t.template st<KE>(r1.y, r);
      }
      t.template st<KE>(r0.y, z);
      t.template keep<KE>(r0.x, r1.w, z);
      break;
    }
    case C_POW: {
      const Vec<T, KE> x = t.template ld<KE>(r0.z), y = t.template ld<KE>(r0.w);
      Vec<T, KE> z;
      NDVM_EACH z.v[j] = pow(x.v[j], y.v[j]);
      t.template st<KE>(r0.y, z);
      t.template keep<KE>(r0.x, r1.w, z);
      break;
    }
    case C_SIN: case C_COS: {
      const Vec<T, KE> x = t.template ld<KE>(r0.z);
      const bool is_sin = (r0.x & 0xff) == C_SIN;
      Vec<T, KE> z;
      if (r1.y != kCNone || (int)r1.z >= 0) {
        Vec<T, KE> w;
        NDVM_EACH {
          T s, c;
          fast_sincos(x.v[j], &s, &c);
          z.v[j] = is_sin ? s : c;
          w.v[j] = is_sin ? c : s;
        }
        if (r1.y != kCNone) t.template st<KE>(r1.y, w);
        if ((int)r1.z >= 0) t.template keep<KE>(kCSave, r1.z, w);
      } else if (is_sin) {
        NDVM_EACH z.v[j] = fast_sin(x.v[j]);
      } else {
        NDVM_EACH z.v[j] = fast_cos(x.v[j]);
      }
      t.template st<KE>(r0.y, z);
      t.template keep<KE>(r0.x, r1.w, z);
      break;
    }
    case C_CMP: {
      const Vec<T, KE> x = t.template ld<KE>(r0.z), y = t.template ld<KE>(r0.w);
      const int k = (r0.x >> kCCountShift) & 7;
      Vec<T, KE> z;
      NDVM_EACH {
        const T p = x.v[j], q = y.v[j];
        const bool r = k == 0 ? p < q : k == 1 ? p <= q : k == 2 ? p > q : k == 3 ? p >= q : p == q;
        z.v[j] = r ? (T)1 : (T)0;
      }
      t.template st<KE>(r0.y, z);
      t.template keep<KE>(r0.x, r1.w, z);
      break;
    }
    case C_SELECT: {
      const Vec<T, KE> p = t.template ld<KE>(r0.z), x = t.template ld<KE>(r0.w), y = t.template ld<KE>(r1.x);
      Vec<T, KE> z;
      NDVM_EACH z.v[j] = !is_zero(p.v[j]) ? x.v[j] : y.v[j];
      t.template st<KE>(r0.y, z);
      t.template keep<KE>(r0.x, r1.w, z);
      break;
    }
    // ------------------------------------------------------------------------ reverse
    case R_DIV: {
      const Vec<T, KE> g = t.template ld<KE>(r0.y), b = t.template ld<KE>(r1.y);
      bool add[KE];
      Vec<T, KE> q;
      if (r1.w != kCNone) {
        const Vec<T, KE> r = t.template ld<KE>(r1.w);
        NDVM_EACH { add[j] = !is_zero(g.v[j]); q.v[j] = (T)0; if (add[j]) q.v[j] = div_by_rcp(g.v[j], b.v[j], r.v[j]); }
      } else {
        NDVM_EACH { add[j] = !is_zero(g.v[j]); q.v[j] = (T)0; if (add[j]) q.v[j] = div_rcp_q(g.v[j], b.v[j]); }
      }
      if (r0.z != kCNone) update<T, K, KE>(t, r0.z, q, add, r0.x & kCFirstA);
      if (r0.w != kCNone) {
        const Vec<T, KE> z = t.template ld<KE>(r1.z);
        NDVM_EACH q.v[j] = -q.v[j];
        update_fma<T, K, KE>(t, r0.w, q, z, add, r0.x & kCFirstB);
      }
      break;
    }
    case R_POW: {
      const Vec<T, KE> g = t.template ld<KE>(r0.y), x = t.template ld<KE>(r1.x), e = t.template ld<KE>(r1.y),
                       z = t.template ld<KE>(r1.z);
      bool add[KE];
      Vec<T, KE> v;
      NDVM_EACH add[j] = !is_zero(g.v[j]);
      if (r0.z != kCNone) {
        NDVM_EACH v.v[j] = g.v[j] * e.v[j] * z.v[j] / x.v[j];
        update<T, K, KE>(t, r0.z, v, add, r0.x & kCFirstA);
      }
      if (r0.w != kCNone) {
        NDVM_EACH v.v[j] = g.v[j] * z.v[j] * log(x.v[j]);
        update<T, K, KE>(t, r0.w, v, add, r0.x & kCFirstB);
      }
      break;
    }
#define NDVM_REV1(OPC, FIELD, EXPR)                               \
  case OPC: {                                                     \
    const Vec<T, KE> gv = t.template ld<KE>(r0.y);                \
    const Vec<T, KE> xv = t.template ld<KE>(FIELD);               \
    bool add[KE];                                                 \
    Vec<T, KE> v;                                                 \
    NDVM_EACH {                                                   \
      const T g = gv.v[j], x = xv.v[j];                           \
      add[j] = !is_zero(g);                                       \
      v.v[j] = (T)0;                                              \
      if (add[j]) v.v[j] = (EXPR);                                \
    }                                                             \
    update<T, K, KE>(t, r0.z, v, add, r0.x & kCFirstA);           \
    break;                                                        \
  }
    NDVM_REV1(R_LOG, r1.x, gt_eps(x) ? div_rcp_q(g, x) : (T)0)
    NDVM_REV1(R_ABS, r1.x, x > (T)0 ? g : (x < (T)0 ? -g : g * (T)0))
#undef NDVM_REV1
    case R_SQRT: {
      const Vec<T, KE> g = t.template ld<KE>(r0.y), x = t.template ld<KE>(r1.x), z = t.template ld<KE>(r1.z);
      bool add[KE];
      Vec<T, KE> v;
      NDVM_EACH {
        add[j] = !is_zero(g.v[j]);
        v.v[j] = (T)0;
        if (add[j] && gt_eps(x.v[j])) v.v[j] = g.v[j] / ((T)2 * z.v[j]);
      }
      update<T, K, KE>(t, r0.z, v, add, r0.x & kCFirstA);
      break;
    }
    case R_TANH: {
      const Vec<T, KE> g = t.template ld<KE>(r0.y), z = t.template ld<KE>(r1.z);
      bool add[KE];
      Vec<T, KE> d;
      NDVM_EACH { add[j] = !is_zero(g.v[j]); d.v[j] = (T)1 - z.v[j] * z.v[j]; }
      update_fma<T, K, KE>(t, r0.z, g, d, add, r0.x & kCFirstA);
      break;
    }
    case R_POWI: {
      const Vec<T, KE> g = t.template ld<KE>(r0.y), x = t.template ld<KE>(r1.x);
      const int n = (int)r1.w;
      bool add[KE];
      Vec<T, KE> d;
      NDVM_EACH { add[j] = !is_zero(g.v[j]); d.v[j] = n > 0 ? powi_deriv(x.v[j], n) : (T)0; }
      update_fma<T, K, KE>(t, r0.z, g, d, add, r0.x & kCFirstA);
      break;
    }
    case R_SELECT: {
      const Vec<T, KE> g = t.template ld<KE>(r0.y), p = t.template ld<KE>(r1.x);
      bool ta[KE], tb[KE];
      NDVM_EACH {
        const bool taken = !is_zero(p.v[j]), on = !is_zero(g.v[j]);
        ta[j] = on && taken;
        tb[j] = on && !taken;
      }
      if (r0.z != kCNone) update<T, K, KE>(t, r0.z, g, ta, r0.x & kCFirstA);
      if (r0.w != kCNone) update<T, K, KE>(t, r0.w, g, tb, r0.x & kCFirstB);
      break;
    }
    case R_DSUM: {
      const Vec<T, KE> g = t.template ld<KE>(r0.y), p = t.template ld<KE>(r1.x);
      bool add[KE];
      NDVM_EACH add[j] = !is_zero(g.v[j]);
      update_fma<T, K, KE>(t, r0.z, g, p, add, r0.x & kCFirstA);
      break;
    }
    default: break;
  }
}

// The same as a call: where the rules are a small part of the stream (long scalar tapes), the
// interpreter's loop then holds fewer registers and its two copies share them.
template <typename T, int K, int KE>
__device__ __noinline__ void rule_call(unsigned base, unsigned save_row, T* save, uint4 r0, uint4 r1) {
  Slots<T, K> t;
  t.base = base;
  t.save_row = save_row;
  t.save = save;
  rule<T, K, KE>(t, r0, r1);
}

// The current points' observations into slots.
template <typename T, int K>
__device__ __forceinline__ void observe(const Thread<T, K>& t, const uint4& r0, const uint4& r1) {
  const int n = (r0.x >> kCCountShift) & 7;
  const uint32_t col[kCCopies] = {r0.z, r1.x, r1.z}, dst[kCCopies] = {r0.y, r0.w, r1.y};
  Vec<T, K> z[kCCopies];
#pragma unroll
  for (int e = 0; e < kCCopies; e++)
    if (e < n) {
#pragma unroll
      for (int j = 0; j < K; j++) z[e].v[j] = t.point[j][col[e]];
    }
#pragma unroll
  for (int e = 0; e < kCCopies; e++)
    if (e < n) t.template st<K>(dst[e], z[e]);
}

// Asynchronous copies of workspace values into slots, and the wait for earlier ones.
template <typename T, int K>
__device__ __forceinline__ void fetch(const Thread<T, K>& t, const uint4& r0, const uint4& r1) {
  const int n = (r0.x >> kCCountShift) & 7;
  const uint32_t src[kCCopies] = {r0.z, r1.x, r1.z}, dst[kCCopies] = {r0.y, r0.w, r1.y};
#pragma unroll
  for (int e = 0; e < kCCopies; e++) {
    if (e >= n) break;
    const unsigned d = t.at(dst[e]);
    const T* s = t.saved(src[e]);
    if (sizeof(T) == 8)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(s) : "memory");
    else
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(s) : "memory");
  }
  if (r0.x & kCCommit) asm volatile("cp.async.commit_group;\n" ::: "memory");
  if (r0.x & kCWait) {  // the thread's own copies: no barrier
    switch ((r0.x >> kCPendingShift) & 7) {
      case 0: asm volatile("cp.async.wait_group 0;\n" ::: "memory"); break;
      case 1: asm volatile("cp.async.wait_group 1;\n" ::: "memory"); break;
      case 2: asm volatile("cp.async.wait_group 2;\n" ::: "memory"); break;
      case 3: asm volatile("cp.async.wait_group 3;\n" ::: "memory"); break;
      default: asm volatile("cp.async.wait_group %0;\n" ::"n"(kFetchWindows) : "memory"); break;
    }
  }
}

// The records at which the inner loop ends and that are not control: loads, sums, results.
template <typename T, int K, int KE>
__device__ __forceinline__ void outer(const Thread<T, K>& t, const uint4& r0, const uint4& r1, const ReplayArgs& a) {
  switch (r0.x & 0xff) {
    // ---------------------------------------------------------------- loads and stores
    case C_LOADC: {
      Vec<T, KE> z;
      const T c = sizeof(T) == 8 ? (T)__hiloint2double((int)r0.w, (int)r0.z) : (T)__uint_as_float(r1.x);
      NDVM_EACH z.v[j] = c;
      t.template st<KE>(r0.y, z);
      break;
    }
    case C_LOADP: case C_LOADO: case C_LOADS: {
      const uint32_t op = r0.x & 0xff;
      const T* src = op == C_LOADP ? t.params + (t.lane * t.P + (int64_t)r0.z)
                   : op == C_LOADO ? t.obs + r0.z
                                   : t.saved(r0.z);
      Vec<T, KE> z;
      const T c = *src;
      NDVM_EACH z.v[j] = c;
      t.template st<KE>(r0.y, z);
      break;
    }
    case C_ZERO: {
      Vec<T, KE> z;
      NDVM_EACH z.v[j] = (T)0;
      for (uint32_t e = 0; e < r0.z; e++) t.template st<KE>(r0.y + e * kCSlotUnit, z);
      break;
    }
    case C_SEED: {
      Vec<T, KE> z;
      NDVM_EACH z.v[j] = (T)1;
      t.template st<KE>(r0.y, z);
      break;
    }
    case C_GREDUCE:
      for (uint32_t e = 0; e < r0.z; e++) {
        const Vec<T, K> p = t.template ld<K>(r0.y + e * kCSlotUnit);
        T s = p.v[0];
#pragma unroll
        for (int j = 1; j < K; j++) s = s + p.v[j];
        for (int o = t.G >> 1; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        Vec<T, KE> z;
        NDVM_EACH z.v[j] = s;
        t.template st<KE>(r0.y + e * kCSlotUnit, z);
      }
      break;
    case C_LOSS:
      if (t.writer) static_cast<T*>(a.loss)[t.lane] = t.template ld<1>(r0.y).v[0];
      break;
    case C_GRAD:
      if (t.writer) static_cast<T*>(a.grad)[t.lane * t.P + r0.z] = r0.y == kCNone ? (T)0 : t.template ld<1>(r0.y).v[0];
      break;
    default:  // not a record of this translation
      if (a.err) atomicExch(a.err, 1);
      break;
  }
}

#undef NDVM_EACH

// One record (words A0, A1; the next record's words go to B0, B1).
#define NDVM_STEP(A0, A1, B0, B1)                                                        \
  {                                                                                      \
    rp += (unsigned)sizeof(CRec);                                                        \
    B0 = ld_words(rp);                                                                   \
    B1 = ld_words(rp + 16);                                                              \
    const uint32_t op = A0.x & 0xff;                                                     \
    if (op == C_ARITH) {                                                                 \
      arith<T, K, KE>(t, A0, A1);                                                        \
    } else if (op >= C_END) {                                                            \
      rp -= (unsigned)sizeof(CRec);                                                      \
      e0 = A0;                                                                           \
      e1 = A1;                                                                           \
      return;                                                                            \
    } else if (K == 1 && op == C_FETCH) {                                                \
      fetch<T, K>(t, A0, A1);                                                            \
    } else if (KE == K && op == C_OBS) {                                                 \
      observe<T, K>(t, A0, A1);                                                          \
    } else {                                                                             \
      if (KE == K && K > 1) rule<T, K, KE>(t, A0, A1);                                   \
      else rule_call<T, K, KE>(t.base, t.save_row, t.save, A0, A1);                      \
    }                                                                                    \
  }

// Runs records from address rp up to the next one that ends the inner loop, whose words it
// returns in e0, e1 (rp then names it).  Each record is read while the one before it runs,
// into the other of two sets of registers.
template <typename T, int K, int KE>
__device__ __forceinline__ void run(const Thread<T, K>& t, unsigned& rp, uint4& e0, uint4& e1) {
  uint4 r0 = ld_words(rp), r1 = ld_words(rp + 16), n0, n1;
  for (;;) {
    NDVM_STEP(r0, r1, n0, n1)
    NDVM_STEP(n0, n1, r0, r1)
  }
}
#undef NDVM_STEP

// CHUNKED: a long loop-free stream in double-buffered chunks of kCChunk records; otherwise
// the whole stream is in shared memory.
template <typename T, int K, bool CHUNKED>
__device__ __forceinline__ void scalar_body(const ReplayArgs& a, const int block) {
  static_assert(!CHUNKED || K == 1, "chunked streams have no loops");
  const int tid = threadIdx.x, tpb = blockDim.x;
  const int64_t lane_raw = a.lane0 + (int64_t)block * (tpb >> a.log2g) + (tid >> a.log2g);
  const unsigned smem = (unsigned)__cvta_generic_to_shared(smem_raw);
  Thread<T, K> t;
  t.G = 1 << a.log2g;
  t.grank = tid & (t.G - 1);
  t.writer = lane_raw < a.lane_end && t.grank == 0;
  t.lane = lane_raw < a.lane_end ? lane_raw : a.lane_end - 1;
  t.save_row = (unsigned)(a.save_ld * (int64_t)sizeof(T));
  t.P = a.P;
  t.obs = static_cast<const T*>(a.obs);
  t.params = static_cast<const T*>(a.params);
  t.save = static_cast<T*>(a.save) + (t.lane - a.lane0);
  t.base = smem + a.stage_off + (unsigned)(tid >> 5) * (unsigned)(a.sstride << (row_shift<T, K>() + 7)) +
           (unsigned)(tid & 31) * (unsigned)(sizeof(T) * K);

  // n records from `first` on into shared memory at dst
  auto stage = [&](int first, int n, unsigned dst) {
    const uint4* src = reinterpret_cast<const uint4*>(a.code) + 2 * (int64_t)first;
    for (int i = tid; i < 2 * n; i += tpb)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 16 * i), "l"(src + i) : "memory");
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  constexpr int kChunkRecs = (int)kCChunk;
  constexpr unsigned kBuf = kCChunk * sizeof(CRec);
  unsigned rp = smem;
  uint4 r0, r1;
  stage(0, CHUNKED ? min(kChunkRecs, a.n_code) : a.n_code, smem);
  if (CHUNKED) {
    for (int first = kChunkRecs, k = 0;; first += kChunkRecs, k++) {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");  // chunk k has landed (and every prefetched value)
      __syncthreads();  // for every thread; and every warp has left chunk k - 1: its buffer is free
      if (first < a.n_code) stage(first, min(kChunkRecs, a.n_code - first), smem + ((k + 1) & 1) * kBuf);
      rp = smem + (k & 1) * kBuf;
      for (;;) {
        run<T, K, 1>(t, rp, r0, r1);
        if ((r0.x & 0xff) <= C_CHUNK) break;
        outer<T, K, 1>(t, r0, r1, a);
        rp += (unsigned)sizeof(CRec);
      }
      if ((r0.x & 0xff) == C_END) return;
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  for (;;) {
    run<T, K, 1>(t, rp, r0, r1);
    if ((r0.x & 0xff) == C_END) return;
    if ((r0.x & 0xff) != C_LOOP) {
      outer<T, K, 1>(t, r0, r1, a);
      rp += (unsigned)sizeof(CRec);
      continue;
    }
    // passes of G x K points: thread grank's points are grank, grank + G, ...
    const int64_t N = r0.y, stride = r0.z, base = r0.w;
    const unsigned end = smem + r1.x * (unsigned)sizeof(CRec), start = rp + (unsigned)sizeof(CRec);
    const uint32_t valid = r1.y;
    const T* from = (r0.x & kCExt) ? reinterpret_cast<const T*>(a.args) : t.obs;
    const int per = t.G * K;
    for (int64_t p0 = 0; p0 < N; p0 += per) {
      Vec<T, K> on;
#pragma unroll
      for (int j = 0; j < K; j++) {
        const int64_t p = p0 + t.grank + (int64_t)j * t.G;
        on.v[j] = p < N ? (T)1 : (T)0;
        t.point[j] = from + (base + (p < N ? p : N - 1) * stride);
      }
      t.template st<K>(valid, on);
      rp = start;
      for (;;) {
        run<T, K, K>(t, rp, r0, r1);
        if ((r0.x & 0xff) == C_ENDLOOP) break;
        outer<T, K, K>(t, r0, r1, a);
        rp += (unsigned)sizeof(CRec);
      }
    }
    rp = end + (unsigned)sizeof(CRec);
  }
}

template <typename T, int K, bool CHUNKED>
__global__ void __launch_bounds__(128, 4) k_scalar(ReplayArgs a) {
  scalar_body<T, K, CHUNKED>(a, blockIdx.x);
}

template <typename T, int K, bool CHUNKED>
__global__ void __launch_bounds__(128, 4) k_scalar_multi(const __grid_constant__ MultiArgs ma) {
  const int b = blockIdx.x;
  int lo = 0, hi = ma.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (ma.start[mid] <= b) lo = mid;
    else hi = mid - 1;
  }
  scalar_body<T, K, CHUNKED>(ma.a[lo], b - ma.start[lo]);
}

// the kernel takes up to `smem` bytes of dynamic shared memory (per device, grown on demand)
template <typename F>
cudaError_t allow_smem(F* kernel, size_t smem, int& dev_done, size_t& smem_done) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev_done == dev && smem <= smem_done) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  dev_done = dev;
  smem_done = smem;
  return cudaSuccess;
}

template <typename T, int K, bool CHUNKED>
cudaError_t launch_one(const ReplayArgs* a, const MultiArgs* m, int blocks, int tpb, size_t smem, cudaStream_t s) {
  static int dev[2] = {-1, -1};
  static size_t done[2] = {0, 0};
  cudaError_t e = m ? allow_smem(k_scalar_multi<T, K, CHUNKED>, smem, dev[1], done[1])
                    : allow_smem(k_scalar<T, K, CHUNKED>, smem, dev[0], done[0]);
  if (e != cudaSuccess) return e;
  if (m) k_scalar_multi<T, K, CHUNKED><<<blocks, tpb, smem, s>>>(*m);
  else k_scalar<T, K, CHUNKED><<<blocks, tpb, smem, s>>>(*a);
  return cudaGetLastError();
}

template <typename T, int KV>
cudaError_t launch_any(const ReplayArgs* a, const MultiArgs* m, int blocks, int tpb, size_t smem, cudaStream_t s) {
  const ReplayArgs& f = m ? m->a[0] : *a;
  if (f.staged) return launch_one<T, 1, true>(a, m, blocks, tpb, smem, s);
  return f.points == 1 ? launch_one<T, 1, false>(a, m, blocks, tpb, smem, s)
                       : launch_one<T, KV, false>(a, m, blocks, tpb, smem, s);
}

}  // namespace

cudaError_t launch_scalar(const ReplayArgs* a, const MultiArgs* m, bool f32, int blocks, int tpb, size_t smem,
                          cudaStream_t s) {
  return f32 ? launch_any<float, kPointsF32>(a, m, blocks, tpb, smem, s)
             : launch_any<double, kPointsF64>(a, m, blocks, tpb, smem, s);
}

}  // namespace ndvm
