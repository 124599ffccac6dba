// Replay of tapes with matrices: an interpreter of matrix records (compact.h), for tapes without
// a data axis.
//
// G consecutive threads of a warp (or block) serve one lane and share its column of slots; they split the elements
// of each matrix result (element e belongs to thread e mod G) and repeat its scalar records.
// What bounds these tapes is the latency of a record where lanes are few (a 4 x 4 product is
// one or two elements per thread: four dependent multiply-adds of 64 cycles, in an interpreter
// that spent 172 instructions per record) and the FP64 pipe where they are many.  So:
//  - every operand of a record is in shared memory, addressed by 32-bit offsets: slots,
//    the program's constant matrices (one copy per block), and workspace values and
//    observations, which are copied into slots of their own kMAhead records before their use;
//  - one record covers a product and, in the other form, both of its adjoint rules, as sums over
//    strided operands; the reverse rules' test for an all-zero adjoint (which contributes nothing, even
//    against an infinite factor) runs only when a sum comes out as NaN;
//  - a product with a constant matrix takes the terms of its nonzero elements only (transition
//    and observation matrices of filters are mostly zeros and ones: 23 % of an 8-state filter's
//    forward work and more of a 4-state one's multiplies by zero).  The result is the same
//    value as long as the other operand is finite: each thread remembers whether it has
//    stored an infinity or a NaN, and a warp in which one has takes every term;
//  - a record's operation word is read from one thread, so that the compiler knows it to be the
//    same in all of them and leaves out the reconvergence around every test of it (a scalar
//    record: 88 -> 75 instructions).
//  - each element loop exists once and is not unrolled: copies per size did not fit in the
//    instruction cache next to each other (the constant-velocity filter below 5.94 -> 5.62).
//  - where a lane's slots leave few warps on an SM, or there are few lanes, a lane has a block of
//    64 to 256 threads (BLOCK), with a barrier of the block after each record.
// Measured on one GB300 against the general kernel (ms): a 4-state constant-velocity filter of 200
// steps, 8192 lanes 6.99 -> 5.62 (FP64 instructions halved), 3001 lanes without gradient 2.78 ->
// 1.96; 256 lanes x 80 steps 2.15 -> 1.75; an 8-state filter of 120 steps, 16384 lanes 23.6 ->
// 19.3; a lane per block: 16 states, 50 lanes x 8 steps 1.24 -> 0.48 and 2000 lanes 1.58 -> 1.34;
// 24 states, 400 lanes x 6 steps 2.12 -> 0.73; 32 states, 1500 lanes x 4 steps 14.2 -> 3.72.
// What binds now is still instructions: about 118 per record, 6 cycles each with one warp
// per scheduler.  Tried and not faster: two elements' chains interleaved (the first filter 7.1), a
// thread's elements in one column with its operand in registers (no change), predicated accesses
// in place of branches, a warp per lane for 12 to 15 states (the same elements, fewer lanes: 12
// states, 8000 lanes x 6 steps 2.83 for 2.34), scaled constant matrices read from global memory
// to save their shared memory (32 states 9 % slower).
#include "interp.cuh"
#include "smallmat.cuh"

namespace ndvm {
namespace {

extern __shared__ __align__(16) unsigned char smem_raw[];

template <typename T>
struct MThread {
  unsigned base;      // shared-memory address of the lane's slot column
  unsigned step;      // bytes from one of the thread's elements to the next: G rows
  unsigned row;       // bytes of a slot row
  unsigned consts;    // address of the constant matrices
  unsigned lists;     // address of the lists of nonzero elements
  unsigned save_row;  // bytes of a workspace row
  const T* obs;
  const T* params;
  T* save;            // the lane's workspace column
  int64_t lane;
  int P, G, g;        // threads per lane, this thread's place among them
  bool writer;

  __device__ __forceinline__ unsigned at(uint32_t slot) const { return base + (slot / kCSlotUnit) * row; }
  template <int KE>
  __device__ __forceinline__ Vec<T, KE> ld(uint32_t slot) const {
    Vec<T, KE> x;
    ld_shared(at(slot), x.v);
    return x;
  }
  // (scalar records: every thread of the lane has the value, one stores it)
  template <int KE>
  __device__ __forceinline__ void st(uint32_t slot, const Vec<T, KE>& x) const {
    if (g == 0) st_shared(at(slot), x.v);
  }
  template <int KE>
  __device__ __forceinline__ void keep(uint32_t flags, uint32_t idx, const Vec<T, KE>& x) const {
    if ((flags & kCSave) && g == 0) *saved(idx) = x.v[0];
  }
  __device__ __forceinline__ T* saved(uint32_t idx) const {
    return reinterpret_cast<T*>(reinterpret_cast<char*>(save) + (uint64_t)idx * save_row);
  }
};

template <typename T>
__device__ __forceinline__ T ld1(unsigned a) {
  T x[1];
  ld_shared(a, x);
  return x[0];
}
template <typename T>
__device__ __forceinline__ void st1(unsigned a, T x) {
  const T v[1] = {x};
  st_shared(a, v);
}
// The high word of |x|: infinities and NaNs are the largest.  (On the bits, off the FP64 pipe.)
__device__ __forceinline__ unsigned size_word(double x) { return (unsigned)(fbits(x) >> 32) & 0x7fffffffu; }
__device__ __forceinline__ unsigned size_word(float x) { return __float_as_uint(x) & 0x7fffffffu; }
template <typename T> constexpr unsigned kInfWord = sizeof(T) == 8 ? 0x7ff00000u : 0x7f800000u;
// the largest high word a thread has stored in a matrix
struct Largest {
  unsigned w = 0;
  template <typename T> __device__ __forceinline__ void see(T x) { w = max(w, size_word(x)); }
};
__device__ __forceinline__ bool is_nan(double x) { return nan_key(abs_key(x), x); }
__device__ __forceinline__ bool is_nan(float x) { return nan_key(abs_key(x), x); }

// address and element stride of a matrix operand
template <typename T>
struct MOperand {
  unsigned a, s;
  __device__ __forceinline__ MOperand(const MThread<T>& t, uint32_t v, bool is_const)
      : a(is_const ? t.consts + v * (unsigned)sizeof(T) : t.at(v)), s(is_const ? (unsigned)sizeof(T) : t.row) {}
  __device__ __forceinline__ T operator[](int e) const { return ld1<T>(a + (unsigned)e * s); }
};

// s + x0 y0 + x1 y1 + ... over K terms, left to right; every load issues before the chain starts
template <typename T, int K>
__device__ __forceinline__ T dot_terms(unsigned x, unsigned xs, unsigned y, unsigned ys, T s) {
  T xv[K], yv[K];
#pragma unroll
  for (int q = 0; q < K; q++) { xv[q] = ld1<T>(x + q * xs); yv[q] = ld1<T>(y + q * ys); }
#pragma unroll
  for (int q = 0; q < K; q++) s = fma(xv[q], yv[q], s);
  return s;
}
// the same over more than 8 terms: even and odd ones in two chains, eight terms' loads at a time
template <typename T>
__device__ __forceinline__ T dot_long(unsigned x, unsigned xs, unsigned y, unsigned ys, int K, T s) {
  T s1 = neg_zero<T>();
  int q = 0;
  for (; q + 8 <= K; q += 8, x += 8 * xs, y += 8 * ys) {
    T xv[8], yv[8];
#pragma unroll
    for (int u = 0; u < 8; u++) { xv[u] = ld1<T>(x + u * xs); yv[u] = ld1<T>(y + u * ys); }
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      s = fma(xv[u], yv[u], s);
      s1 = fma(xv[u + 1], yv[u + 1], s1);
    }
  }
  for (; q + 1 < K; q += 2, x += 2 * xs, y += 2 * ys) {
    s = fma(ld1<T>(x), ld1<T>(y), s);
    s1 = fma(ld1<T>(x + xs), ld1<T>(y + ys), s1);
  }
  if (q < K) s = fma(ld1<T>(x), ld1<T>(y), s);
  return s + s1;
}

template <typename T>
__device__ __noinline__ bool all_zero_at(unsigned a, unsigned s, int n) {
#pragma unroll 1
  for (int e = 0; e < n; e++)
    if (!is_zero(ld1<T>(a + (unsigned)e * s))) return false;
  return true;
}

// The words of the frequent records as the kernel reads them: once per block and chunk, decode()
// turns slots and element strides into byte offsets and strides (an operand's offset is from the
// lane's column, or, for a constant, an address).
//   w1 result, w2 X, w3 Y, w4 elements; and for products: w5 xi, w6 xq,
//   w7 save, w8 2^20 / cols, w9 yq, w10 yj, w11 and w12 result and operand of the sum that follows,
//   w13 its save, w14 elements of the gating operand | NZ << 13 | cols << 20, w15 list address | K << 24
template <typename T>
__device__ void decode(const ReplayArgs& a, unsigned rp, unsigned consts, unsigned lists) {
  const uint4 r0 = ld_words(rp), r1 = ld_words(rp + 16), r2 = ld_words(rp + 32), r3 = ld_words(rp + 48);
  const unsigned row = (unsigned)a.sstride * (unsigned)sizeof(T), size = (unsigned)sizeof(T);
  auto off = [&](uint32_t slot) { return slot == kCNone ? kCNone : slot / kCSlotUnit * row; };
  auto operand = [&](uint32_t v, bool c) { return c ? consts + v * size : off(v); };
  auto put = [&](unsigned at, uint4 v) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w));
  };
  const uint32_t op = r0.x & 0xff, f = r0.x;
  if (op == C_ARITH) {
    put(rp, make_uint4(f, off(r0.y), off(r0.z), off(r0.w)));
    put(rp + 16, make_uint4(off(r1.x), r1.y, r1.z, r1.w));
  } else if (op >= M_F && op <= M_RSELECT) {
    const bool cx = f & kMConstX, cy = f & kMConstY;
    const unsigned xs = cx ? size : row, ys = cy ? size : row;
    const unsigned rows = r1.x & 0xff, cols = (r1.x >> 8) & 0xff, K = (r1.x >> 16) & 0xff, NZ = r1.x >> 24;
    put(rp, make_uint4(f, off(r0.y), operand(r0.z, cx), operand(r0.w, cy)));
    put(rp + 16, make_uint4(rows * cols, (r1.y & 0xffff) * xs, (r1.y >> 16) * xs, r1.w));
    put(rp + 32, make_uint4(r2.y, (r1.z & 0xffff) * ys, (r1.z >> 16) * ys, off(r2.w)));
    put(rp + 48, make_uint4((f & kMPost) ? operand(r3.x, f & kMPostConst) : 0u, r3.y, r2.z | NZ << 13 | cols << 20,
                            (lists + 4u * r2.x) | K << 24));
  } else if (op == M_ADD || op == M_COPY) {
    put(rp, make_uint4(f, off(r0.y), off(r0.z), off(r0.w)));
  } else if (op == M_FETCH) {
    put(rp, make_uint4(f, off(r0.y), r0.z, r0.w));
  }
}

// A product's record: where it starts element e's sum, and what it does with it.  REV: an
// adjoint's product (gates, accumulates, subtracts); else a forward one (saves, and the sum or
// difference that follows).
template <typename T, bool REV>
struct Product {
  const MThread<T>& t;
  uint32_t f;
  unsigned out;
  uint4 r0, r1, r2, r3;

  __device__ __forceinline__ Product(const MThread<T>& th, unsigned rp, const uint4& w0, const uint4& w1) : t(th), r0(w0), r1(w1) {
    f = r0.x;
    out = t.base + r0.y;
    r2 = ld_words(rp + 32);
    r3 = ld_words(rp + 48);
  }
  __device__ __forceinline__ int cols() const { return (int)(r3.z >> 20); }
  // element e's sum starts at; on: e is an element and the thread's
  __device__ __forceinline__ T start(unsigned o) const {
    T s = neg_zero<T>();
    if (REV && (f & kMAcc)) s = with_sign(ld1<T>(out + o), f);
    return s;
  }
  __device__ __forceinline__ void finish(int e, unsigned o, bool on, T s, T z, Largest& bad) const {
    bad.see(z);
    if (REV) {
      if (size_word(z) >= kInfWord<T> && (f & (kMGateX | kMGateY)) && is_nan(z) &&
          all_zero_at<T>(t.base + ((f & kMGateX) ? r0.z : r0.w), t.row, (int)(r3.z & 0x1fffu)))
        z = (f & kMAcc) ? s : (T)0;
      if (on) st1<T>(out + o, with_sign(z, f));
    } else {
      if (on) st1<T>(out + o, z);
      if (f & kCSave) {
        if (on) *t.saved(r1.w + (unsigned)e) = z;
      }
      if (f & kMPost) {
        const T c = ld1<T>((f & kMPostConst) ? r3.x + (unsigned)e * (unsigned)sizeof(T) : t.base + r3.x + o);
        const T y = c + with_sign(z, (f & kMPostNeg) ? 0x80000000u : 0u);
        bad.see(y);
        if (on) {
          st1<T>(t.base + r2.w + o, y);
          if ((int)r3.y >= 0) *t.saved(r3.y + (unsigned)e) = y;
        }
      }
    }
  }
};

// The thread's elements of n: every thread of the warp makes the same passes; one without an
// element in the last pass repeats the result's last element and does not store it (on = false).
// (One copy of the body, not unrolled: the interpreter's code is larger than the instruction
// cache, and two copies or unrolled loops cost the 8-state filter 10 %.)
template <typename T, typename F>
__device__ __forceinline__ void each_element(const MThread<T>& t, int n, F f) {
  int e = t.g;
  unsigned o = (unsigned)t.g * t.row;
#pragma unroll 1
  do {
    const bool on = e < n;
    const int c = on ? e : n - 1;
    f(c, on ? o : (unsigned)c * t.row, on);
    e += t.G;
    o += t.step;
  } while (e - t.g < n);
}

// The thread's elements of a product over K terms (K = 0: more than 8).
template <typename T, int K, bool REV>
__device__ __forceinline__ void dense(const MThread<T>& t, unsigned rp, const uint4& r0, const uint4& r1, Largest& bad) {
  const Product<T, REV> p(t, rp, r0, r1);
  const int cols = p.cols();
  const unsigned X = p.r0.z + ((p.f & kMConstX) ? 0u : t.base), Y = p.r0.w + ((p.f & kMConstY) ? 0u : t.base);
  each_element(t, (int)r1.x, [&](int e, unsigned o, bool on) {
    const int i = (int)(((uint32_t)e * p.r2.x) >> 20), j = e - i * cols;
    const unsigned x = X + (unsigned)i * p.r1.y, y = Y + (unsigned)j * p.r2.z;
    const T s = p.start(o);
    T z;
    if constexpr (K > 0) z = dot_terms<T, K>(x, p.r1.z, y, p.r2.y, s);
    else z = dot_long<T>(x, p.r1.z, y, p.r2.y, (int)(p.r3.w >> 24), s);
    p.finish(e, o, on, s, z, bad);
  });
}

__device__ __forceinline__ uint32_t ld_word(unsigned a) {
  uint32_t q;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(q) : "r"(a));
  return q;
}

// A product with a list: every term if its warp has met an infinity or a NaN (all); else the list's
// terms in two chains (kMChains: sums over more than 8).  A call: in the loop of sparse below the test
// for the second chain costs the small filters 3 to 6 %.
template <typename T, bool REV>
__device__ __noinline__ unsigned list_call(MThread<T> t, unsigned rp, uint4 r0, uint4 r1, bool all) {
  Largest bad;
  const Product<T, REV> p(t, rp, r0, r1);
  const unsigned X = p.r0.z + ((p.f & kMConstX) ? 0u : t.base), Y = p.r0.w + ((p.f & kMConstY) ? 0u : t.base);
  const int K = (int)(p.r3.w >> 24);
  each_element(t, (int)r1.x, [&](int e, unsigned o, bool on) {
    const int i = (int)(((uint32_t)e * p.r2.x) >> 20), j = e - i * p.cols();
    unsigned x = X + (unsigned)i * p.r1.y, y = Y + (unsigned)j * p.r2.z;
    const T s = p.start(o);
    T z = s;
    if (!all) {
      const int NZ = (int)((p.r3.z >> 13) & 0x7fu);
      const uint32_t v = (p.f & kMOtherY) ? r0.w : r0.z;
      const bool both = (p.f & kMConstX) && (p.f & kMConstY);
      const unsigned other = both ? v : t.base + v, step = both ? (unsigned)sizeof(T) : t.row;
      const unsigned l = (p.r3.w & 0xffffffu) + 4u * (unsigned)(e * NZ);
      T odd = neg_zero<T>();
      bool second = false;
#pragma unroll 1
      for (int u = 0; u < NZ; u++) {
        const uint32_t q = ld_word(l + 4u * (unsigned)u);
        if (q == kCNone) break;
        if (q == kMSplit) { second = true; continue; }
        const T c = ld1<T>(t.consts + (q & 0xffffu) * (unsigned)sizeof(T)), w = ld1<T>(other + (q >> 16) * step);
        if (second) odd = fma(c, w, odd);
        else z = fma(c, w, z);
      }
      z = z + odd;
      if (!(p.f & kMAcc) && is_zero(z)) z = (T)0;  // (as in sparse)
    } else if (K > 8) {
      z = dot_long<T>(x, p.r1.z, y, p.r2.y, K, s);
    } else {
      for (int q = 0; q < K; q++, x += p.r1.z, y += p.r2.y) z = fma(ld1<T>(x), ld1<T>(y), z);
    }
    p.finish(e, o, on, s, z, bad);
  });
  return bad.w;
}

// M_FSPARSE, M_RSPARSE: the terms of the constant operand's nonzero elements
template <typename T, bool REV>
__device__ __forceinline__ void sparse(const MThread<T>& t, unsigned rp, const uint4& r0, const uint4& r1, Largest& bad) {
  const Product<T, REV> p(t, rp, r0, r1);
  const int NZ = (int)((p.r3.z >> 13) & 0x7fu);
  const uint32_t v = (p.f & kMOtherY) ? r0.w : r0.z;
  const bool both = (p.f & kMConstX) && (p.f & kMConstY);
  const unsigned other = both ? v : t.base + v, step = both ? (unsigned)sizeof(T) : t.row;
  each_element(t, (int)r1.x, [&](int e, unsigned o, bool on) {
    const unsigned l = (p.r3.w & 0xffffffu) + 4u * (unsigned)(e * NZ);
    const T s = p.start(o);
    T z = s;
#pragma unroll 1
    for (int u = 0; u < NZ; u++) {
      const uint32_t q = ld_word(l + 4u * (unsigned)u);
      if (q == kCNone) break;
      z = fma(ld1<T>(t.consts + (q & 0xffffu) * (unsigned)sizeof(T)), ld1<T>(other + (q >> 16) * step), z);
    }
    if (!(p.f & kMAcc) && is_zero(z)) z = (T)0;  // the terms left out are zeros: -0 only if all were
    p.finish(e, o, on, s, z, bad);
  });
}

// M_SELECT, M_RSELECT: elements of slots, by a list
template <typename T, bool REV>
__device__ __forceinline__ void select(const MThread<T>& t, unsigned rp, const uint4& r0, const uint4& r1, Largest& bad) {
  const Product<T, REV> p(t, rp, r0, r1);
  const unsigned other = t.base + ((p.f & kMOtherY) ? r0.w : r0.z), list = p.r3.w & 0xffffffu;
  each_element(t, (int)r1.x, [&](int e, unsigned o, bool on) {
    const uint32_t q = ld_word(list + 4u * (unsigned)e);
    T z = ld1<T>(other + (q == kCNone ? 0u : q) * t.row);
    if (q == kCNone) z = (T)0;
    p.finish(e, o, on, neg_zero<T>(), z, bad);
  });
}

// M_ADD, M_COPY
template <typename T, bool COPY>
__device__ __forceinline__ void add(const MThread<T>& t, const uint4& r0, const uint4& r1, Largest& bad) {
  const unsigned out = t.base + r0.y, a = t.base + r0.z, b = t.base + r0.w;
  each_element(t, (int)r1.x, [&](int e, unsigned o, bool on) {
    T z;
    if (COPY) z = with_sign(ld1<T>(a + o), r0.x);
    else z = ld1<T>(a + o) + with_sign(ld1<T>(b + o), r0.x);
    bad.see(z);
    if (on) {
      st1<T>(out + o, z);
      if (r0.x & kCSave) *t.saved(r1.w + (unsigned)e) = z;
    }
  });
}

// C_ARITH (decoded)
template <typename T>
__device__ __forceinline__ void arith_decoded(const MThread<T>& t, const uint4& r0, const uint4& r1) {
  const T x = ld1<T>(t.base + r0.z), y = ld1<T>(t.base + r0.w), c = ld1<T>(t.base + r1.x);
  const bool off = (r0.x & kCGate) && is_zero(x);
  const T z = fma(with_sign(x, r0.x), off ? (T)0 : y, c);
  if (t.g == 0) st1<T>(t.base + r0.y, z);
  if (r0.x & kCSave) {
    if (t.g == 0) *t.saved(r1.w) = z;
  }
}

// what gauss_jordan asks of a lane (pointers into shared memory)
template <typename T>
struct GjLane {
  T* sbase;
  int ss, eg, es;
  __device__ __forceinline__ T* wp(int32_t slot) const { return sbase + slot * ss; }
  __device__ __forceinline__ int first() const { return eg; }
  __device__ __forceinline__ int step() const { return es; }
};

// M_INV, M_DET, M_LOGDET
template <typename T>
__device__ __noinline__ unsigned small_matrix(MThread<T> t, unsigned smem0, uint4 r0, uint4 r1) {
  const uint32_t op = r0.x & 0xff;
  const int n = (int)(r1.x & 0xffu);
  const uint32_t mn = r1.x >> 8;
  GjLane<T> L;
  L.sbase = reinterpret_cast<T*>(smem_raw + (t.base - smem0));
  L.ss = (int)(t.row / sizeof(T));
  L.eg = t.g;
  L.es = min(t.G, 32);  // (a lane over several warps: the first one)
  const Opnd<T> A = {L.wp((int)(r0.z / kCSlotUnit)), L.ss};
  const int scratch = (int)(r0.w / kCSlotUnit);
  const bool inverse = op == M_INV || r1.y != kCNone || (int)r1.z >= 0;
  uint32_t perm = 0;
  T det = (T)0, r = (T)0;
  Largest bad;
  if (n <= 3) {
    det = det_small(A, n);
    if (inverse) r = rcp_rn(det);
  } else {
    det = gauss_jordan<T, true>(L, A, n, scratch, inverse, perm);
  }
  if (op != M_INV) {
    Vec<T, 1> z;
    z.v[0] = op == M_DET ? det : fast_log(det);
    t.template st<1>(r0.y, z);
    t.template keep<1>(r0.x, r1.w, z);
  }
  if (inverse) {
    const uint32_t out = op == M_INV ? r0.y : r1.y;
    const int sv = op == M_INV ? ((r0.x & kCSave) ? (int)r1.w : -1) : (int)r1.z;
    for (int e = t.g; e < n * n; e += L.es) {
      const T v = n <= 3 ? inv_small(A, n, e, r) : gj_inverse<T>(L, scratch, n, perm, (int)(((uint32_t)e * mn) >> 20), e - (int)(((uint32_t)e * mn) >> 20) * n);
      bad.see(v);
      if (out != kCNone) st1<T>(t.at(out) + (unsigned)e * t.row, v);
      if (sv >= 0) *t.saved((unsigned)(sv + e)) = v;
    }
  }
  return bad.w;
}

// value of an element named by an operand reference of the argument lists
template <typename T>
__device__ __forceinline__ T element(const MThread<T>& t, const ReplayArgs& a, int32_t ref) {
  const uint32_t kind = ((uint32_t)ref >> 28) & 7u;
  const int32_t idx = ref & kRefIndexMask;
  if (kind == RK_SLOT) return ld1<T>(t.base + (unsigned)idx * t.row);
  if (kind == RK_CONST) return static_cast<const T*>(a.consts)[idx];
  if (kind == RK_OBS) return t.obs[idx];
  if (kind == RK_SAVE) return *t.saved((unsigned)idx);
  return t.params[t.lane * t.P + idx];
}

template <typename T>
__device__ __forceinline__ void zero_own(const MThread<T>& t, unsigned at, int n) {
  for (int e = t.g; e < n; e += t.G) st1<T>(at + (unsigned)e * t.row, (T)0);
}

// The matrix records besides products and small inverses.
template <typename T>
__device__ __forceinline__ void matrix_rule(const MThread<T>& t, const uint4& r0, const uint4& r1, const ReplayArgs& a,
                                            bool finite, Largest& bad) {
  const uint32_t f = r0.x;
  const bool fa = f & kCFirstA, fb = f & kCFirstB;
  switch (f & 0xff) {
    case M_ADDC: {
      const MOperand<T> A(t, r0.z, f & kMConstX), B(t, r0.w, f & kMConstY);
      const unsigned out = t.at(r0.y);
#pragma unroll 1
      for (int e = t.g; e < (int)r1.x; e += t.G) {
        const T z = A[e] + with_sign(B[e], f);
        bad.see(z);
        st1<T>(out + (unsigned)e * t.row, z);
        if (f & kCSave) *t.saved(r1.w + (unsigned)e) = z;
      }
      break;
    }
    case M_SCALE: {
      const T s = MOperand<T>(t, r0.z, f & kMConstX)[0];
      const MOperand<T> A(t, r0.w, f & kMConstY);
      const unsigned out = t.at(r0.y);
#pragma unroll 1
      for (int e = t.g; e < (int)r1.x; e += t.G) {
        const T z = s * A[e];
        bad.see(z);
        st1<T>(out + (unsigned)e * t.row, z);
        if (f & kCSave) *t.saved(r1.w + (unsigned)e) = z;
      }
      break;
    }
    case M_TRACE: {
      const MOperand<T> A(t, r0.z, f & kMConstX);
      const int n = (int)r1.x;
      Vec<T, 1> s;
      s.v[0] = A[0];
      for (int i = 1; i < n; i++) s.v[0] = s.v[0] + A[i * n + i];
      t.template st<1>(r0.y, s);
      t.template keep<1>(f, r1.w, s);
      break;
    }
    case M_GATHER: {
      const unsigned out = t.at(r0.y);
#pragma unroll 1
      for (int e = t.g; e < (int)r0.w; e += t.G) {
        const T z = element<T>(t, a, a.args[r0.z + (unsigned)e]);
        bad.see(z);
        st1<T>(out + (unsigned)e * t.row, z);
        if (f & kCSave) *t.saved(r1.w + (unsigned)e) = z;
      }
      break;
    }
    case M_FETCH: {  // (a thread copies the elements that it stored)
      const unsigned out = t.base + r0.y;
#pragma unroll 1
      for (int e = t.g; e < (int)r0.w; e += t.G) {
        const T* src = (f & kMFromObs) ? t.obs + (r0.z + (unsigned)e) : t.saved(r0.z + (unsigned)e);
        if (sizeof(T) == 8)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(out + (unsigned)e * t.row), "l"(src) : "memory");
        else
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(out + (unsigned)e * t.row), "l"(src) : "memory");
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
      break;
    }
    case M_RSCALE: {
      const unsigned g = t.at(r0.y);
      const int w = (int)r1.x;
      const bool zero = all_zero_at<T>(g, t.row, w);
      if (r0.z != kCNone) {
        Vec<T, 1> s;
        s.v[0] = fa ? neg_zero<T>() : t.template ld<1>(r0.z).v[0];
        if (zero) {
          if (fa) s.v[0] = (T)0;
        } else {
          // (a constant's zeros add nothing to a finite sum; a lane over several warps: the first one)
          const MOperand<T> A(t, r1.z, f & kMConstY);
          const bool skip = finite && (f & kMConstY);
          if (t.g < 32)
#pragma unroll 1
            for (int e = 0; e < w; e++) {
              const T x = A[e];
              if (!skip || !is_zero(x)) s.v[0] = fma(ld1<T>(g + (unsigned)e * t.row), x, s.v[0]);
            }
        }
        t.template st<1>(r0.z, s);
      }
      if (r0.w != kCNone) {
        const unsigned o = t.at(r0.w);
        if (zero) {
          if (fb) zero_own(t, o, w);
        } else {
          const T s = MOperand<T>(t, r1.y, f & kMConstX)[0];
    #pragma unroll 1
      for (int e = t.g; e < w; e += t.G) {
            const unsigned q = o + (unsigned)e * t.row;
            const T z = fma(s, ld1<T>(g + (unsigned)e * t.row), fb ? neg_zero<T>() : ld1<T>(q));
            bad.see(z);
            st1<T>(q, z);
          }
        }
      }
      break;
    }
    case M_RDET: {
      const int n = (int)(r1.x & 0xffu);
      const T g = t.template ld<1>(r0.y).v[0];
      const unsigned o = t.at(r0.z);
      if (is_zero(g)) {
        if (fa) zero_own(t, o, n * n);
        break;
      }
      const T fac = r1.y != kCNone ? g * t.template ld<1>(r1.y).v[0] : g;
      const MOperand<T> I(t, r1.z, false);
      const uint32_t mn = r1.x >> 8;
#pragma unroll 1
      for (int e = t.g; e < n * n; e += t.G) {
        const int i = (int)(((uint32_t)e * mn) >> 20), j = e - i * n;
        const unsigned q = o + (unsigned)e * t.row;
        const T z = fma(fac, I[j * n + i], fa ? neg_zero<T>() : ld1<T>(q));
        bad.see(z);
        st1<T>(q, z);
      }
      break;
    }
    case M_RTRACE: {
      const int n = (int)r1.x;
      const T g = t.template ld<1>(r0.y).v[0];
      const unsigned o = t.at(r0.z);
      if (fa) zero_own(t, o, n * n);
      if (is_zero(g)) break;
      for (int i = 0; i < n; i++) {
        const int e = i * n + i;
        if ((e & (t.G - 1)) != t.g) continue;
        const T z = ld1<T>(o + (unsigned)e * t.row) + g;
        bad.see(z);
        st1<T>(o + (unsigned)e * t.row, z);
      }
      break;
    }
    case M_RGATHER: {
      // (targets are scalars; one may be named several times: in order, one thread)
      const unsigned g = t.at(r0.y);
      const bool zero = all_zero_at<T>(g, t.row, (int)r0.w);
      if (t.g == 0)
        for (int e = 0; e < (int)r0.w; e++) {
          const int32_t target = a.args[r0.z + 2 * (unsigned)e];
          if (target == -1) continue;
          const bool first = a.args[r0.z + 2 * (unsigned)e + 1] != 0;
          const unsigned q = t.base + (unsigned)(target & kRefIndexMask) * t.row;
          if (zero) {
            if (first) st1<T>(q, (T)0);
          } else {
            const T v = ld1<T>(g + (unsigned)e * t.row);
            st1<T>(q, first ? v : ld1<T>(q) + v);
          }
        }
      break;
    }
    case M_RSCATTER: {
      const unsigned g = t.at(r0.y), o = t.at(r0.z);
      if (fa) zero_own(t, o, (int)r1.y);
      for (int e = 0; e < (int)r1.x; e++) {
        const int m = a.args[r0.w + (unsigned)e];
        if ((m & (t.G - 1)) != t.g) continue;
        const T z = ld1<T>(o + (unsigned)m * t.row) + ld1<T>(g + (unsigned)e * t.row);
        bad.see(z);
        st1<T>(o + (unsigned)m * t.row, z);
      }
      break;
    }
    default:  // not a record of this translation
      if (a.err) atomicExch(a.err, 1);
      break;
  }
}

template <typename T>
__device__ __noinline__ void scalar_rule(MThread<T> t, uint4 r0, uint4 r1) { rule<T, 1>(t, r0, r1); }

// BLOCK: a lane has the whole block, G = 64 to 256 threads (large matrices, few lanes): a block
// barrier after every record, scalar records and small inverses in the first warp.
template <typename T, bool BLOCK>
__device__ __forceinline__ void matrix_body(const ReplayArgs& a, const int block) {
  const int tid = threadIdx.x, tpb = blockDim.x;
  const unsigned smem = (unsigned)__cvta_generic_to_shared(smem_raw);
  const int64_t lane_raw = a.lane0 + (int64_t)block * (tpb >> a.log2g) + (tid >> a.log2g);
  constexpr unsigned kBuf = kMChunk * sizeof(MRec);
  constexpr int kChunkRecs = (int)kMChunk;
  const unsigned const_bytes = ((unsigned)a.n_consts * (unsigned)sizeof(T) + 15u) & ~15u;
  const unsigned list_bytes = ((unsigned)a.n_lists * 4u + 15u) & ~15u;
  MThread<T> t;
  t.G = 1 << a.log2g;
  t.g = tid & (t.G - 1);
  t.writer = lane_raw < a.lane_end && t.g == 0;
  t.lane = lane_raw < a.lane_end ? lane_raw : a.lane_end - 1;
  t.P = a.P;
  t.obs = static_cast<const T*>(a.obs);
  t.params = static_cast<const T*>(a.params);
  t.save = static_cast<T*>(a.save) + (t.lane - a.lane0);
  t.save_row = (unsigned)(a.save_ld * (int64_t)sizeof(T));
  t.row = (unsigned)a.sstride * (unsigned)sizeof(T);
  t.consts = smem + 2 * kBuf;
  t.lists = t.consts + const_bytes;
  t.base = smem + (unsigned)a.stage_off + (unsigned)(tid >> a.log2g) * (unsigned)sizeof(T);

  t.step = (unsigned)t.G * t.row;

  const uint4* code = reinterpret_cast<const uint4*>(a.code);
  auto copy = [&](const uint4* src, unsigned dst, int pieces) {
    for (int i = tid; i < pieces; i += tpb)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 16 * i), "l"(src + i) : "memory");
  };
  auto stage = [&](int first, unsigned dst) {
    copy(code + 4 * (int64_t)first, dst, 4 * min(kChunkRecs, a.n_code - first));
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  copy(code + 4 * (int64_t)a.n_code, t.consts, (int)((const_bytes + list_bytes) / 16));
  stage(0, smem);
  Largest bad;
  // whether a thread of the warp (or block) has stored an infinity or a NaN
  auto met = [&]() -> bool {
    if (BLOCK) return __syncthreads_or(bad.w >= kInfWord<T>);
    return __any_sync(0xffffffffu, bad.w >= kInfWord<T>);
  };
  for (int first = kChunkRecs, k = 0;; first += kChunkRecs, k++) {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");  // chunk k has landed (and every staged operand)
    __syncthreads();  // for every thread; and every warp has left chunk k - 1: its buffer is free
    if (first < a.n_code) stage(first, smem + ((k + 1) & 1) * kBuf);
    unsigned rp = smem + (k & 1) * kBuf;
    for (int r = tid; r < min(kChunkRecs, a.n_code - (first - kChunkRecs)); r += tpb)
      decode<T>(a, rp + (unsigned)r * (unsigned)sizeof(MRec), t.consts, t.lists);
    __syncthreads();
    for (;; rp += (unsigned)sizeof(MRec)) {
      uint4 r0 = ld_words(rp);
      uint4 r1 = ld_words(rp + 16);
      // (the same in every thread; from one of them, the compiler knows it to be)
      r0.x = __shfl_sync(0xffffffffu, r0.x, 0);
      r1.x = __shfl_sync(0xffffffffu, r1.x, 0);
      const uint32_t op = r0.x & 0xff;
#define NDVM_DENSE(K)                                                      \
  case M_F + K: dense<T, K, false>(t, rp, r0, r1, bad); break;            \
  case M_R + K: dense<T, K, true>(t, rp, r0, r1, bad); break;
      const bool others = BLOCK && tid >= 32 && ((op < M_F && op != C_FETCH && op != C_CHUNK && op != C_END) ||
                                                 (op >= M_INV && op <= M_TRACE));
      if (!others) switch (op) {  // (else the first warp's record)
        case C_ARITH: arith_decoded<T>(t, r0, r1); break;
        NDVM_DENSE(0) NDVM_DENSE(1) NDVM_DENSE(2) NDVM_DENSE(3) NDVM_DENSE(4) NDVM_DENSE(5) NDVM_DENSE(6)
        NDVM_DENSE(7) NDVM_DENSE(8)
        case M_FSPARSE:
          if (const bool all = met(); all || (r0.x & kMChains)) bad.w = max(bad.w, list_call<T, false>(t, rp, r0, r1, all));
          else sparse<T, false>(t, rp, r0, r1, bad);
          break;
        case M_RSPARSE:
          if (const bool all = met(); all || (r0.x & kMChains)) bad.w = max(bad.w, list_call<T, true>(t, rp, r0, r1, all));
          else sparse<T, true>(t, rp, r0, r1, bad);
          break;
        case M_SELECT:  // (without a constant operand: a gather, not a product)
          if ((r0.x & (kMConstX | kMConstY)) && met()) bad.w = max(bad.w, list_call<T, false>(t, rp, r0, r1, true));
          else select<T, false>(t, rp, r0, r1, bad);
          break;
        case M_RSELECT:
          if ((r0.x & (kMConstX | kMConstY)) && met()) bad.w = max(bad.w, list_call<T, true>(t, rp, r0, r1, true));
          else select<T, true>(t, rp, r0, r1, bad);
          break;
        case M_ADD: add<T, false>(t, r0, r1, bad); break;
        case M_COPY: add<T, true>(t, r0, r1, bad); break;
        case C_FETCH: fetch<T>(t, r0, r1, t.g == 0); break;
        case M_INV: case M_DET: case M_LOGDET: bad.w = max(bad.w, small_matrix<T>(t, smem, r0, r1)); break;
        case C_CHUNK: goto next_chunk;
        case C_END: return;
        default:
          if (op > M_F) matrix_rule<T>(t, r0, r1, a, op == M_RSCALE && !met(), bad);
          else if (op < C_END) scalar_rule<T>(t, r0, r1);
          else outer<T, 1, 1>(t, r0, r1, a);
      }
#undef NDVM_DENSE
      const uint32_t wait = (r0.x >> kMWaitShift) & 7u;
      if (wait) {  // the next record reads copied operands
        if (wait == 1) asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        else asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      }
      // the lane's threads see each other's elements
      if (BLOCK) __syncthreads();
      else __syncwarp();
    }
  next_chunk:;
  }
}

template <typename T, bool BLOCK>
__global__ void __launch_bounds__(BLOCK ? 256 : 128, BLOCK ? 2 : 4) k_matrix(ReplayArgs a) {
  matrix_body<T, BLOCK>(a, blockIdx.x);
}

template <typename T, bool BLOCK>
__global__ void __launch_bounds__(BLOCK ? 256 : 128, BLOCK ? 2 : 4) k_matrix_multi(const __grid_constant__ MultiArgs ma) {
  const int b = blockIdx.x;
  int lo = 0, hi = ma.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (ma.start[mid] <= b) lo = mid;
    else hi = mid - 1;
  }
  matrix_body<T, BLOCK>(ma.a[lo], b - ma.start[lo]);
}

template <typename T, bool BLOCK>
cudaError_t launch(const ReplayArgs* a, const MultiArgs* m, int blocks, int tpb, size_t smem, cudaStream_t s) {
  static SmemLimit one, many;
  cudaError_t e = m ? many.allow(k_matrix_multi<T, BLOCK>, smem) : one.allow(k_matrix<T, BLOCK>, smem);
  if (e != cudaSuccess) return e;
  if (m) k_matrix_multi<T, BLOCK><<<blocks, tpb, smem, s>>>(*m);
  else k_matrix<T, BLOCK><<<blocks, tpb, smem, s>>>(*a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_type(const ReplayArgs* a, const MultiArgs* m, int blocks, int tpb, size_t smem, cudaStream_t s) {
  return (m ? m->a[0] : *a).log2g > 5 ? launch<T, true>(a, m, blocks, tpb, smem, s)
                                      : launch<T, false>(a, m, blocks, tpb, smem, s);
}

}  // namespace

cudaError_t launch_matrix(const ReplayArgs* a, const MultiArgs* m, bool f32, int blocks, int tpb, size_t smem,
                          cudaStream_t s) {
  return f32 ? launch_type<float>(a, m, blocks, tpb, smem, s) : launch_type<double>(a, m, blocks, tpb, smem, s);
}

}  // namespace ndvm
