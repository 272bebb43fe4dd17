// Jacobi building blocks shared by the eigensolvers (eig.cu, eig_dense.cu).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace fpca_jacobi {

// Integers that order as the numbers do, NaN below all (and 64-bit comparisons are slow here).
__device__ __forceinline__ int eig_key(float x) {
  const int b = __float_as_int(x);
  if (isnan(x)) return (int)0x80000000;
  return b >= 0 ? b : (b << 1) == 0 ? 0 : b ^ 0x7fffffff;
}
__device__ __forceinline__ long long eig_key(double x) {
  const long long b = __double_as_longlong(x), m = b & 0x7fffffffffffffffll;
  if (m > 0x7ff0000000000000ll) return (long long)0x8000000000000000ull;
  return b >= 0 ? b : m == 0 ? 0 : b ^ 0x7fffffffffffffffll;
}

// The eigenvalue of key a (place i) comes before that of key b (place j): descending, ties by
// place, NaN last.  A total order, so that ranks are a permutation and every rank's entry is
// written.
template <typename K>
__device__ __forceinline__ bool eig_before(K a, int i, K b, int j) {
  static_assert(std::is_integral<K>::value, "keys");
  return a > b || (a == b && i < j);
}

// The dense eigensolvers work on A 2^-e, e the exponent for which the largest entry lies in
// [1/2, 1): their FP32 copies, squares and thresholds then neither overflow nor vanish whatever
// the scale of the data (from 1.8e19 on a square of FP32 is infinite), and the scaling is exact.
// `top`: the bits of the largest |entry|, which order as the numbers do; not finite: e = 0.
constexpr unsigned long long EIG_INF = 0x7ff0000000000000ull;
__device__ __forceinline__ int eig_exponent(unsigned long long top) {
  if (top == 0 || top >= EIG_INF) return 0;
  return ilogb(__longlong_as_double((long long)top)) + 1;
}
// x 2^-e, by the exponent bits where both are normal numbers (FP64 operations are slow here)
__device__ __forceinline__ double eig_scaled(double x, int e) {
  const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
  if (ex > 0 && ex < 0x7ff && ex - e > 0 && ex - e < 0x7ff)
    return __hiloint2double(hi - e * (1 << 20), __double2loint(x));
  return scalbn(x, -e);
}

// Pair (p, q), p < q, of position i (0 <= i < ne / 2) at step `step` of a sweep of
// the round-robin (circle) schedule: ne / 2 disjoint pairs per step, ne - 1 steps
// (ne even; q == n marks the dummy of odd n).
__device__ __forceinline__ void rr_pair(int ne, int step, int i, int& p, int& q) {
  const int m = ne - 1;
  if (i == 0) {
    p = m;
    q = step;
  } else {
    p = step + i;
    if (p >= m) p -= m;
    q = step - i;
    if (q < 0) q += m;
  }
  if (p > q) {
    const int t = p;
    p = q;
    q = t;
  }
}

// The rotation (c, s) that annihilates a_pq: tau = (a_qq - a_pp) / (2 a_pq),
// t = sign(tau) / (|tau| + sqrt(1 + tau^2)), c = 1 / sqrt(1 + t^2), s = t c.
// Approximate reciprocals and square roots (each gives 0 for an infinite tau^2): a serial
// chain of rotations waits on them, c^2 + s^2 = 1 holds to a few FP32 ulps all the same, and
// the refinement that follows every FP32 Jacobi restores orthogonality.
__device__ __forceinline__ void bj_rot(float app, float apq, float aqq, float& c, float& sn) {
  const float tau = __fdividef(aqq - app, 2.f * apq);
  float root;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(root) : "f"(fmaf(tau, tau, 1.f)));
  const float t = __fdividef(copysignf(1.f, tau), fabsf(tau) + root);
  const bool on = fabsf(apq) > 1e-30f && fabsf(apq) > 1e-18f * fmaxf(fabsf(app), fabsf(aqq));
  c = on ? rsqrtf(fmaf(t, t, 1.f)) : 1.f;
  sn = on ? t * c : 0.f;
}

// The same from the matrix A (n x n, leading dimension ld); q >= n: none.
__device__ __forceinline__ void rr_rot(const float* A, int ld, int n, int p, int q, float& c,
                                       float& sn) {
  if (q < n) {
    bj_rot(A[p * ld + p], A[p * ld + q], A[q * ld + q], c, sn);
  } else {
    c = 1.f;
    sn = 0.f;
  }
}

// ---------------------------------------------------------------------------
// block Jacobi (dense symmetric eigensolver)
// ---------------------------------------------------------------------------
constexpr int BJ_S = 16;        // indices per block
constexpr int BJ_W = 2 * BJ_S;  // subproblem width
constexpr int BJ_NT = 256;      // threads of a subproblem sweep: one per 2 x 2 block
constexpr int BJ_LD = 48;       // leading dimension of a subproblem in shared memory

// local index i of the subproblem of block pair (I, J) -> global index
__device__ __forceinline__ int bj_index(int I, int J, int i) {
  return i < BJ_S ? I * BJ_S + i : J * BJ_S + (i - BJ_S);
}

// The 16 disjoint pairs of step s of a subproblem sweep: `within` (s = 0..14) the pairs
// inside either block, otherwise (s = 0..15) the pairs across the two blocks.
__device__ __forceinline__ void bj_step_pair(bool within, int s, int i, int& p, int& q) {
  if (within) {
    rr_pair(BJ_S, s, i & 7, p, q);
    p += (i >> 3) * BJ_S;
    q += (i >> 3) * BJ_S;
  } else {
    p = i;
    q = BJ_S + ((i + s) & (BJ_S - 1));
  }
}

// One sweep of rotations over the 32 x 32 subproblem in `cur` (leading dimension BJ_LD,
// double-buffered with `nxt`), accumulated into J (32 x 32, leading dimension ldj, identity on
// entry).  The pairs across the blocks meet once; those inside a block only when `within` is
// set (once per sweep of the whole matrix is enough, since each block takes part in every
// round).  A serial chain of 16 or 31 steps, so each of the 256 threads forms the two rotations
// of its 2 x 2 block itself and a step has one barrier; the J entries of the pairs across the
// blocks stay in registers, the column that a pair gives up going to the next lane.  BJ_LD: the
// two rows of a warp in different banks.  (Sixteen threads forming a step's rotations for all,
// with exact square roots, took 0.47 us a step: see k_bj_cluster.)
__device__ __forceinline__ void bj_sweep(float* cur, float* nxt, float* J, int ldj, bool within) {
  constexpr int ld = BJ_LD;
  const int bi = threadIdx.x >> 4, bj = threadIdx.x & 15;
  float cj, sj;
  auto turn = [&](int pi, int qi, int pj, int qj) {
    float ci, si;
    bj_rot(cur[pi * ld + pi], cur[pi * ld + qi], cur[qi * ld + qi], ci, si);
    bj_rot(cur[pj * ld + pj], cur[pj * ld + qj], cur[qj * ld + qj], cj, sj);
    const float m00 = cur[pi * ld + pj], m01 = cur[pi * ld + qj];
    const float m10 = cur[qi * ld + pj], m11 = cur[qi * ld + qj];
    const float c00 = cj * m00 - sj * m01, c01 = sj * m00 + cj * m01;
    const float c10 = cj * m10 - sj * m11, c11 = sj * m10 + cj * m11;
    nxt[pi * ld + pj] = ci * c00 - si * c10;
    nxt[pi * ld + qj] = ci * c01 - si * c11;
    nxt[qi * ld + pj] = si * c00 + ci * c10;
    nxt[qi * ld + qj] = si * c01 + ci * c11;
    float* t = cur;
    cur = nxt;
    nxt = t;
  };
  if (within) {
    for (int s = 0; s < BJ_S - 1; ++s) {
      int pi, qi, pj, qj;
      bj_step_pair(true, s, bi, pi, qi);
      bj_step_pair(true, s, bj, pj, qj);
      turn(pi, qi, pj, qj);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float* row = J + (bi + 16 * h) * ldj;
        const float vp = row[pj], vq = row[qj];
        row[pj] = cj * vp - sj * vq;
        row[qj] = sj * vp + cj * vq;
      }
      __syncthreads();
    }
  }
  float vp[2], vq[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    vp[h] = J[(bi + 16 * h) * ldj + bj];
    vq[h] = J[(bi + 16 * h) * ldj + BJ_S + bj];
  }
  const int next = (threadIdx.x & 16) | ((bj + 1) & 15);
#pragma unroll 4
  for (int s = 0; s < BJ_S; ++s) {
    turn(bi, BJ_S + ((bi + s) & (BJ_S - 1)), bj, BJ_S + ((bj + s) & (BJ_S - 1)));
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float a = vp[h], b = vq[h];
      vp[h] = cj * a - sj * b;
      vq[h] = __shfl_sync(0xffffffffu, sj * a + cj * b, next);
    }
    __syncthreads();
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    J[(bi + 16 * h) * ldj + bj] = vp[h];
    J[(bi + 16 * h) * ldj + BJ_S + bj] = vq[h];
  }
  __syncthreads();
}

}  // namespace fpca_jacobi
