// Device code of the compact-record interpreters (scalar.cu, matrix.cu): shared-memory access
// by 32-bit addresses and the scalar records' arithmetic.  The slot type S of a function says
// where a slot lies: ld, st (a vector of KE values of a slot), keep and saved (workspace).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "compact.h"
#include "replay.h"
#include "rules.cuh"

namespace ndvm {
namespace {

template <typename T, int K>
struct alignas(sizeof(T) * K) Vec {
  T v[K];
};

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

// x + y behind a call: an addition predicated on a flag would take its FP64 slot either way
template <typename T> __device__ __noinline__ T add_call(T x, T y) { return x + y; }

__device__ __forceinline__ double with_sign(double x, uint32_t sign) {  // x, negated when sign's top bit is set
  return __hiloint2double(__double2hiint(x) ^ (int)(sign & 0x80000000u), __double2loint(x));
}
__device__ __forceinline__ float with_sign(float x, uint32_t sign) {
  return __uint_as_float(__float_as_uint(x) ^ (sign & 0x80000000u));
}

// target += v[j] where add[j] (a first contribution stores; where not add[j] it stores 0)
template <typename T, int KE, typename S>
__device__ __forceinline__ void update(const S& t, uint32_t target, const Vec<T, KE>& v, const bool* add, bool first) {
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
template <typename T, int KE, typename S>
__device__ __forceinline__ void update_fma(const S& t, uint32_t target, const Vec<T, KE>& a, const Vec<T, KE>& b,
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
template <typename T, int KE, typename S>
__device__ __forceinline__ void arith(const S& t, const uint4& r0, const uint4& r1) {
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
template <typename T, int KE, typename S>
__device__ __forceinline__ void rule(const S& t, const uint4& r0, const uint4& r1) {
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
      if (r0.z != kCNone) update<T, KE>(t, r0.z, q, add, r0.x & kCFirstA);
      if (r0.w != kCNone) {
        const Vec<T, KE> z = t.template ld<KE>(r1.z);
        NDVM_EACH q.v[j] = -q.v[j];
        update_fma<T, KE>(t, r0.w, q, z, add, r0.x & kCFirstB);
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
        update<T, KE>(t, r0.z, v, add, r0.x & kCFirstA);
      }
      if (r0.w != kCNone) {
        NDVM_EACH v.v[j] = g.v[j] * z.v[j] * log(x.v[j]);
        update<T, KE>(t, r0.w, v, add, r0.x & kCFirstB);
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
    update<T, KE>(t, r0.z, v, add, r0.x & kCFirstA);           \
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
      update<T, KE>(t, r0.z, v, add, r0.x & kCFirstA);
      break;
    }
    case R_TANH: {
      const Vec<T, KE> g = t.template ld<KE>(r0.y), z = t.template ld<KE>(r1.z);
      bool add[KE];
      Vec<T, KE> d;
      NDVM_EACH { add[j] = !is_zero(g.v[j]); d.v[j] = (T)1 - z.v[j] * z.v[j]; }
      update_fma<T, KE>(t, r0.z, g, d, add, r0.x & kCFirstA);
      break;
    }
    case R_POWI: {
      const Vec<T, KE> g = t.template ld<KE>(r0.y), x = t.template ld<KE>(r1.x);
      const int n = (int)r1.w;
      bool add[KE];
      Vec<T, KE> d;
      NDVM_EACH { add[j] = !is_zero(g.v[j]); d.v[j] = n > 0 ? powi_deriv(x.v[j], n) : (T)0; }
      update_fma<T, KE>(t, r0.z, g, d, add, r0.x & kCFirstA);
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
      if (r0.z != kCNone) update<T, KE>(t, r0.z, g, ta, r0.x & kCFirstA);
      if (r0.w != kCNone) update<T, KE>(t, r0.w, g, tb, r0.x & kCFirstB);
      break;
    }
    case R_DSUM: {
      const Vec<T, KE> g = t.template ld<KE>(r0.y), p = t.template ld<KE>(r1.x);
      bool add[KE];
      NDVM_EACH add[j] = !is_zero(g.v[j]);
      update_fma<T, KE>(t, r0.z, g, p, add, r0.x & kCFirstA);
      break;
    }
    default: break;
  }
}

// Asynchronous copies of workspace values into slots (by the threads that `copy`), and the wait
// for earlier ones.
template <typename T, typename S>
__device__ __forceinline__ void fetch(const S& t, const uint4& r0, const uint4& r1, bool copy) {
  const int n = copy ? (int)((r0.x >> kCCountShift) & 7) : 0;
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
template <typename T, int K, int KE, typename S>
__device__ __forceinline__ void outer(const S& t, const uint4& r0, const uint4& r1, const ReplayArgs& a) {
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

// The dynamic shared memory a kernel has been allowed on a device, raised on demand.
class SmemLimit {
 public:
  template <typename F>
  cudaError_t allow(F* kernel, size_t smem) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev_ == dev && smem <= smem_) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    dev_ = dev;
    smem_ = smem;
    return cudaSuccess;
  }

 private:
  int dev_ = -1;
  size_t smem_ = 0;
};

}  // namespace
}  // namespace ndvm
