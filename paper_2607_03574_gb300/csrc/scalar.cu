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
// binary64 on 8 streams, 2.65 -> 2.14 (the FP64 pipe; fmath.cuh's shorter functions are 0.16 of
// it).  Tried and slower on the logistic tape:
// two records per dispatch, independent or with the second reading the first's result from
// a register (2.23 binary64), no reading ahead of the next record (2.48), and record kinds of
// their own for gated or saved arithmetic (2.14).
#include "interp.cuh"

namespace ndvm {
namespace {

extern __shared__ __align__(16) unsigned char smem_raw[];

// log2 of a slot row (32 threads x K values) in units of kCSlotUnit
template <typename T, int K>
__host__ __device__ constexpr int row_shift() {
  return (sizeof(T) * K == 4) ? 0 : (sizeof(T) * K == 8) ? 1 : 2;
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

// The same as a call: where the rules are a small part of the stream (long scalar tapes), the
// interpreter's loop then holds fewer registers and its two copies share them.
template <typename T, int K, int KE>
__device__ __noinline__ void rule_call(unsigned base, unsigned save_row, T* save, uint4 r0, uint4 r1) {
  Slots<T, K> t;
  t.base = base;
  t.save_row = save_row;
  t.save = save;
  rule<T, KE>(t, r0, r1);
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

// One record (words A0, A1; the next record's words go to B0, B1).
#define NDVM_STEP(A0, A1, B0, B1)                                                        \
  {                                                                                      \
    rp += (unsigned)sizeof(CRec);                                                        \
    B0 = ld_words(rp);                                                                   \
    B1 = ld_words(rp + 16);                                                              \
    const uint32_t op = A0.x & 0xff;                                                     \
    if (op == C_ARITH) {                                                                 \
      arith<T, KE>(t, A0, A1)   ;                                                        \
    } else if (op >= C_END) {                                                            \
      rp -= (unsigned)sizeof(CRec);                                                      \
      e0 = A0;                                                                           \
      e1 = A1;                                                                           \
      return;                                                                            \
    } else if (K == 1 && op == C_FETCH) {                                                \
      fetch<T>(t, A0, A1, true);                                                            \
    } else if (KE == K && op == C_OBS) {                                                 \
      observe<T, K>(t, A0, A1);                                                          \
    } else {                                                                             \
      if (KE == K && K > 1) rule<T, KE>(t, A0, A1);                                      \
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

template <typename T, int K, bool CHUNKED>
cudaError_t launch_one(const ReplayArgs* a, const MultiArgs* m, int blocks, int tpb, size_t smem, cudaStream_t s) {
  static SmemLimit one, many;
  cudaError_t e = m ? many.allow(k_scalar_multi<T, K, CHUNKED>, smem) : one.allow(k_scalar<T, K, CHUNKED>, smem);
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
