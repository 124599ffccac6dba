// Small-matrix arithmetic of the replay kernels: closed forms to 3 x 3, Gauss-Jordan elimination
// split over a lane's threads to 8 x 8.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "rules.cuh"

namespace ndvm {
namespace {

// operand view: element e is p[e * s] (the host keeps e * s within 32 bits)
template <typename T>
struct Opnd {
  const T* p;
  int s;
  __device__ __forceinline__ T operator[](int e) const { return p[e * s]; }
  __device__ __forceinline__ const T* at(int e) const { return p + e * s; }
};

// Determinants and inverses to 3 x 3 in closed form, element by element: a lane's
// thread group splits an inverse's elements like those of any other matrix result,
// and every element has the same arithmetic whichever thread computes it.
// cofactor of element (r, s) of a 3 x 3 matrix (the cyclic form carries the sign)
template <typename T>
__device__ __forceinline__ T cof3(const Opnd<T>& A, int r, int s) {
  const int r1 = r == 2 ? 0 : r + 1, r2 = r == 0 ? 2 : r - 1;
  const int s1 = s == 2 ? 0 : s + 1, s2 = s == 0 ? 2 : s - 1;
  return fma(A[r1 * 3 + s1], A[r2 * 3 + s2], -(A[r1 * 3 + s2] * A[r2 * 3 + s1]));
}
// determinant, n <= 3 (expansion along the first row)
template <typename T>
__device__ __forceinline__ T det_small(const Opnd<T>& A, int n) {
  if (n == 1) return A[0];
  if (n == 2) return fma(A[0], A[3], -(A[1] * A[2]));
  return fma(A[2], cof3(A, 0, 2), fma(A[1], cof3(A, 0, 1), A[0] * cof3(A, 0, 0)));
}
// element e of the inverse, n <= 3, given r = 1 / det: the adjugate's element times r
template <typename T>
__device__ __forceinline__ T inv_small(const Opnd<T>& A, int n, int e, T r) {
  if (n == 1) return r;
  if (n == 2) return flip_sign(A[(e == 0 || e == 3) ? 3 - e : e], (unsigned)(e == 1 || e == 2)) * r;
  const int i = e / 3, j = e - 3 * i;
  return cof3(A, j, i) * r;
}

// IEEE bits of |x| as an integer: ordered like |x| for every value that is not a NaN
__device__ __forceinline__ unsigned long long abs_key(double x) {
  return (unsigned long long)fbits(x) & 0x7fffffffffffffffULL;
}
__device__ __forceinline__ unsigned long long abs_key(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ bool nan_key(unsigned long long k, double) { return k > 0x7ff0000000000000ULL; }
__device__ __forceinline__ bool nan_key(unsigned long long k, float) { return k > 0x7f800000ULL; }

// Gauss-Jordan elimination with partial pivoting (n = 4..8) on [A | I] (want_inv) or on
// A alone, in the lane's scratch slots at sref: n rows of wc = 2n (or n) elements,
// row-major.  Rows are never moved: the exchanges are kept as a permutation in a
// register, four bits per logical row, logical row i being physical row perm(i).  The
// lane's threads split the columns: in a column step a thread normalizes the pivot row
// in its own columns and eliminates the other rows there, so the only values the
// threads share within a step are the pivot column's, which every thread reads before
// any is written.  The pivot is the first logical row at or below the diagonal of
// largest magnitude (a strict comparison; a NaN never wins), a row whose factor is
// exactly zero is left alone, and every element takes the same operations as in the
// sequential elimination.  Returns the determinant (the product of the pivots, negated
// per exchange); the inverse's row i is physical row perm(i), columns n .. 2n-1.
template <typename T, bool SYNC, typename LaneT>
__device__ T gauss_jordan(const LaneT& L, const Opnd<T>& A, int n, int32_t sref, bool want_inv, uint32_t& perm) {
  T* W = L.wp(sref);
  const int ss = L.ss, wc = want_inv ? 2 * n : n;
  const int first = L.first(), es = L.step();
  for (int j = first; j < wc; j += es)
    for (int i = 0; i < n; i++) W[(i * wc + j) * ss] = j < n ? A[i * n + j] : (T)(j - n == i ? 1 : 0);
  perm = 0x76543210u;
  if (SYNC) __syncwarp();
  T d = (T)1;
  for (int col = 0; col < n; col++) {
    int piv = col;
    unsigned long long best = abs_key(W[((int)((perm >> (4 * col)) & 15u) * wc + col) * ss]);
    for (int i = col + 1; i < n; i++) {
      const unsigned long long k = abs_key(W[((int)((perm >> (4 * i)) & 15u) * wc + col) * ss]);
      if (!nan_key(k, T()) && !nan_key(best, T()) && k > best) { best = k; piv = i; }
    }
    if (piv != col) {
      const uint32_t a = (perm >> (4 * col)) & 15u, b = (perm >> (4 * piv)) & 15u;
      perm = (perm & ~((15u << (4 * col)) | (15u << (4 * piv)))) | (b << (4 * col)) | (a << (4 * piv));
      d = -d;
    }
    const int pr = (int)((perm >> (4 * col)) & 15u);
    const T pv = W[(pr * wc + col) * ss];
    d = d * pv;
    const T r = rcp_rn(pv);
    T fct[8];  // the pivot column in the other rows, by physical row
#pragma unroll
    for (int i = 0; i < 8; i++) fct[i] = (i < n && i != pr) ? W[(i * wc + col) * ss] : (T)0;
    if (SYNC) __syncwarp();
    for (int j = first; j < wc; j += es) {
      const T p = W[(pr * wc + j) * ss] * r;
      W[(pr * wc + j) * ss] = p;
#pragma unroll
      for (int i = 0; i < 8; i++)
        if (i < n && i != pr && !is_zero(fct[i])) W[(i * wc + j) * ss] = fma(-fct[i], p, W[(i * wc + j) * ss]);
    }
    if (SYNC) __syncwarp();
  }
  return d;
}
// element (i, j) of the inverse left by gauss_jordan in the scratch slots
template <typename T, typename LaneT>
__device__ __forceinline__ T gj_inverse(const LaneT& L, int32_t sref, int n, uint32_t perm, int i, int j) {
  return L.wp(sref)[((int)((perm >> (4 * i)) & 15u) * 2 * n + n + j) * L.ss];
}

}  // namespace
}  // namespace ndvm
