// Leading eigenpairs of a symmetric FP64 matrix with n <= 256 (the dense path of
// fpca_rproj_eig on small grids).
//
// A serial chain bounds it: some 75 rounds of dependent rotations at 256 x 256 (1.2 ms; 2.6
// with two barriers and exact square roots in a rotation step, and sweeps until every
// off-diagonal was small).  The whole FP64 fit of a 16 x 16 grid takes 1.3 to 1.4 ms with it and
// took 4.9 ms through launch_dense_eig (180 launches of each round's two kernels among them);
// of a 64-node curve 0.43 ms, from 1.16.
//
//  1. Block Jacobi in FP32 on one thread-block cluster (k_bj_cluster): all eigenvectors to
//     about 1e-5 or better, or until the off-diagonal norm is LE_APART of the wanted gaps.
//  2. The k leading vectors (and a few more, so that nearly equal eigenvalues at the edge
//     are ordered by their refined values) are refined in FP64 against the FP32 basis X:
//     for vector x_j,  s_ij = x_i' A x_j,  r_ij = delta_ij - x_i' x_j,
//     lambda_j = s_jj / (1 - r_jj),  e_ij = (s_ij + lambda_j r_ij) / (lambda_j - lambda_i)
//     (r_ij / 2 within a cluster),  x_j <- x_j + sum_i x_i e_ij: the columns j of the
//     refinement of Ogita and Aishima ("Iterative refinement for symmetric eigenvalue
//     decomposition", 2018).  With only these columns renewed an iteration multiplies their
//     error by the basis' own (1e-5 or better over the relative gap) instead of squaring it,
//     and costs 3 n^2 k FP64 multiply-adds instead of 4 n^3: FP64 runs at 1/64 of the FP32
//     rate here, and refining all n vectors took 0.47 ms of 256 x 256.
//     All of it works on a matrix scaled to entries below 1 (eig_exponent).
//  3. Where this leaves a wanted vector unconverged (eigenvalues closer than the FP32
//     couplings of the basis, a null space), the basis is made orthonormal in FP64 and
//     X'AX, nearly diagonal, diagonalised by FP64 Jacobi (k_lead_full, k_rotate; both
//     return at once otherwise).
#include <cooperative_groups.h>

#include <algorithm>

#include "fpca_internal.cuh"
#include "jacobi.cuh"

namespace cg = cooperative_groups;

namespace {

using namespace fpca_jacobi;

constexpr int LE_MAXN = 256;    // 8 block pairs: a portable cluster of 8 CTAs
constexpr int LE_SWEEPS = 12;
constexpr int LE_EXTRA = 4;     // vectors refined beyond k
constexpr int LE_ITERS = 8;
constexpr float LE_APART = 0.02f;  // off-diagonal norm over the gap that the refinement is left
constexpr int LE_JLD = BJ_W + 4;             // row stride of a J in shared memory (16-byte rows)
constexpr int LE_JS = BJ_W * LE_JLD + 4;     // floats per J: the 4 shift the banks of the next

inline int le_ne(int n) { return (n + BJ_W - 1) / BJ_W * BJ_W; }
__host__ __device__ constexpr int le_ld(int ne) { return ne + ne / 4; }

inline size_t le_smem(int ne) {
  return sizeof(float) * (2 * (size_t)BJ_W * le_ld(ne) + (size_t)BJ_W * ne +
                          (size_t)(ne / BJ_W) * LE_JS + 2 * BJ_W * BJ_LD + LE_MAXN + 16 + 16);
}

// Two-sided block Jacobi, one CTA per block pair of a round, the CTAs of the matrix in one
// cluster.  Per round CTA a reads the 32 rows of its pair from A (L2-resident, 256 KB at
// most), sweeps its 32 x 32 subproblem, hands its rotation J_a to every CTA through
// distributed shared memory, and writes its rows of J' A J back; its 32 rows of V stay in
// its shared memory for the whole run.  The cluster barrier (two per round) stands in for
// the two launches per round of the large-n path.  Columns of the row tiles are stored in
// groups of 16 spaced by 20 floats, so that eight blocks' columns fall in different banks.
__global__ void __launch_bounds__(BJ_NT, 1)
    k_bj_cluster(int n, int ne, int lead, int kk, const double* __restrict__ A64, float* __restrict__ A,
                 double* __restrict__ X, double* __restrict__ X0, float* __restrict__ lam32,
                 int* __restrict__ nref) {
  extern __shared__ __align__(16) float bjc[];
  const cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), NC = (int)cl.num_blocks();
  const int nb = ne / BJ_S, LD = le_ld(ne), tid = threadIdx.x;
  float* Ar = bjc;                        // [32][LD]
  float* Vr = Ar + BJ_W * LD;             // [32][LD]
  float* T = Vr + BJ_W * LD;              // [32][ne]
  float* Jall = T + BJ_W * ne;            // [NC][LE_JS]
  float* a0 = Jall + NC * LE_JS;          // [32][BJ_LD]
  float* a1 = a0 + BJ_W * BJ_LD;
  float* dg = a1 + BJ_W * BJ_LD;          // [256]: the diagonal after a sweep
  float* mass = dg + LE_MAXN;             // [8][2]: every CTA's off-diagonal, diagonal mass
  float* red = mass + 16;                 // [8][2]
  for (int e = tid; e < BJ_W * ne; e += BJ_NT) {
    const int i = e / ne, c = e - i * ne, gi = rank * BJ_W + i;
    __stcg(A + (size_t)gi * ne + c, (gi < n && c < n) ? (float)A64[(size_t)gi * n + c] : 0.f);
    Vr[i * LD + c + 4 * (c >> 4)] = gi == c ? 1.f : 0.f;
  }
  cl.sync();
  // the products' tile of this thread: rows 4 rg.., 8 columns (threads beyond ne idle)
  const bool act = tid < ne;
  const int ncg = ne / 8, rg = act ? tid / ncg : 0, cgp = act ? tid - rg * ncg : 0;
  float prev = 3e38f;
  int done = 0;
  for (int sweep = 0; sweep < LE_SWEEPS; ++sweep) {
    for (int r = 0; r < nb - 1; ++r) {
      int I, J;
      rr_pair(nb, r, rank, I, J);
#pragma unroll 4
      for (int e = tid; e < BJ_W * (ne / 4); e += BJ_NT) {
        const int i = e / (ne / 4), c4 = e - i * (ne / 4);
        *reinterpret_cast<float4*>(Ar + i * LD + 4 * c4 + 4 * (c4 >> 2)) =
            __ldcg(reinterpret_cast<const float4*>(A + (size_t)bj_index(I, J, i) * ne) + c4);
      }
      float* Jl = Jall + rank * LE_JS;
      __syncthreads();
      for (int e = tid; e < BJ_W * BJ_W; e += BJ_NT) {
        const int i = e / BJ_W, j = e % BJ_W;
        a0[i * BJ_LD + j] = Ar[i * LD + (j < BJ_S ? 20 * I + j : 20 * J + j - BJ_S)];
        Jl[i * LE_JLD + j] = i == j ? 1.f : 0.f;
      }
      __syncthreads();
      bj_sweep(a0, a1, Jl, LE_JLD, r == 0);
      for (int c = 0; c < NC; ++c) {
        if (c == rank) continue;
        float4* dst = reinterpret_cast<float4*>(cl.map_shared_rank(Jall, c) + rank * LE_JS);
        for (int e = tid; e < BJ_W * LE_JLD / 4; e += BJ_NT)
          dst[e] = reinterpret_cast<const float4*>(Jl)[e];
      }
      cl.sync();
      // T = A[P_a, :] J (columns grouped by pair) and V <- V J
      float t[4][8], v[4][8];
      int Ib = 0, Jb = 0;
      const int b = cgp >> 2, jj = (cgp & 3) * 8;
      if (act) {
        rr_pair(nb, r, b, Ib, Jb);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int x = 0; x < 8; ++x) t[q][x] = v[q][x] = 0.f;
        const float* jr = Jall + b * LE_JS + jj;
        for (int h = 0; h < 2; ++h) {
          const float* ac = Ar + 4 * rg * LD + 20 * (h ? Jb : Ib);
          const float* vc = Vr + 4 * rg * LD + 20 * (h ? Jb : Ib);
#pragma unroll 1
          for (int k = 0; k < BJ_S; k += 4) {
            float a[4][4], w[4][4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float4 av = *reinterpret_cast<const float4*>(ac + q * LD + k);
              const float4 wv = *reinterpret_cast<const float4*>(vc + q * LD + k);
              a[q][0] = av.x, a[q][1] = av.y, a[q][2] = av.z, a[q][3] = av.w;
              w[q][0] = wv.x, w[q][1] = wv.y, w[q][2] = wv.z, w[q][3] = wv.w;
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              const float* jp = jr + (h * BJ_S + k + kk) * LE_JLD;
              const float4 j0 = *reinterpret_cast<const float4*>(jp);
              const float4 j1 = *reinterpret_cast<const float4*>(jp + 4);
              const float jv[8] = {j0.x, j0.y, j0.z, j0.w, j1.x, j1.y, j1.z, j1.w};
#pragma unroll
              for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                  t[q][x] = fmaf(a[q][kk], jv[x], t[q][x]);
                  v[q][x] = fmaf(w[q][kk], jv[x], v[q][x]);
                }
            }
          }
        }
      }
      __syncthreads();  // V is read above and overwritten in place
      if (act) {
        const int vp = jj < BJ_S ? 20 * Ib + jj : 20 * Jb + jj - BJ_S;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float4* tr = reinterpret_cast<float4*>(T + (4 * rg + q) * ne + 8 * cgp);
          tr[0] = make_float4(t[q][0], t[q][1], t[q][2], t[q][3]);
          tr[1] = make_float4(t[q][4], t[q][5], t[q][6], t[q][7]);
          float4* vr = reinterpret_cast<float4*>(Vr + (4 * rg + q) * LD + vp);
          vr[0] = make_float4(v[q][0], v[q][1], v[q][2], v[q][3]);
          vr[1] = make_float4(v[q][4], v[q][5], v[q][6], v[q][7]);
        }
      }
      __syncthreads();
      // rows of J_a' T, written to their natural places in A
      float off = 0.f, dia = 0.f;
      if (act) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int x = 0; x < 8; ++x) t[q][x] = 0.f;
        const float* ja = Jl + 4 * rg;
        const float* tc = T + 4 * cgp;
#pragma unroll 8
        for (int k = 0; k < BJ_W; ++k) {
          const float4 a = *reinterpret_cast<const float4*>(ja + k * LE_JLD);
          const float4 t0 = *reinterpret_cast<const float4*>(tc + k * ne);
          const float4 t1 = *reinterpret_cast<const float4*>(tc + k * ne + ne / 2);
          const float av[4] = {a.x, a.y, a.z, a.w};
          const float tv[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int x = 0; x < 8; ++x) t[q][x] = fmaf(av[q], tv[x], t[q][x]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int gc = 4 * cgp + h * (ne / 2);  // grouped column -> pair, natural column
          int I2, J2;
          rr_pair(nb, r, gc >> 5, I2, J2);
          const int col = bj_index(I2, J2, gc & 31);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int row = bj_index(I, J, 4 * rg + q);
            const float* o = t[q] + 4 * h;
            __stcg(reinterpret_cast<float4*>(A + (size_t)row * ne + col),
                   make_float4(o[0], o[1], o[2], o[3]));
#pragma unroll
            for (int x = 0; x < 4; ++x) {
              if (row == col + x) dia += o[x] * o[x];
              else off += o[x] * o[x];
            }
          }
        }
      }
      if (r == nb - 2) {
        for (int o = 16; o > 0; o >>= 1) {
          off += __shfl_xor_sync(0xffffffffu, off, o);
          dia += __shfl_xor_sync(0xffffffffu, dia, o);
        }
        if ((tid & 31) == 0) {
          red[2 * (tid >> 5)] = off;
          red[2 * (tid >> 5) + 1] = dia;
        }
        __syncthreads();
        if (tid < 2 * NC) {  // sum tid & 1 of this CTA to CTA tid / 2
          float sum = 0.f;
          for (int w = 0; w < BJ_NT / 32; ++w) sum += red[2 * w + (tid & 1)];
          cl.map_shared_rank(mass, tid >> 1)[2 * rank + (tid & 1)] = sum;
        }
      }
      cl.sync();
    }
    // the same sums in the same order in every CTA: a uniform decision
    float off = 0.f, dia = 0.f;
    for (int c = 0; c < NC; ++c) {
      off += mass[2 * c];
      dia += mass[2 * c + 1];
    }
    // converged to an off-diagonal norm of 1e-5 of the diagonal's, or stalled below 1e-4
    if (off <= 1e-10f * dia || off == 0.f || (off <= 1e-8f * dia && off > 0.25f * prev)) break;
    prev = off;
    // or the `lead` largest eigenvalues stand so far from all others that the refinement takes
    // the rest: what is left of the off-diagonal bounds every eigenvalue's error (Weyl) and,
    // over the nearest gap, the factor by which an iteration there shrinks the error.  Only
    // those are refined then (*nref): the others may still be mixed with one another.
    if (off <= 1e-4f * dia) {
      __syncthreads();
      if (tid < n) dg[tid] = __ldcg(A + (size_t)tid * ne + tid);
      __syncthreads();
      bool apart = true;
      if (tid < n) {
        const float d = dg[tid];
        float gap = 3e38f;
        int rank = 0;
        for (int j = 0; j < n; ++j) {
          rank += dg[j] > d || (dg[j] == d && j < tid);
          if (j != tid) gap = fminf(gap, fabsf(dg[j] - d));
        }
        apart = rank >= lead || sqrtf(off) <= LE_APART * gap;
      }
      done = __syncthreads_and(apart);
      if (done) break;
    }
  }
  for (int e = tid; e < BJ_W * n; e += BJ_NT) {
    const int i = e / n, c = e - i * n, gi = rank * BJ_W + i;
    if (gi < n) {
      const double v = (double)Vr[i * LD + c + 4 * (c >> 4)];
      X[(size_t)gi * n + c] = v;   // refined columns are written over here
      X0[(size_t)gi * n + c] = v;  // the fall-back's basis
    }
  }
  if (rank == 0 && tid == 0) *nref = done ? lead : kk;
  if (tid < BJ_W && rank * BJ_W + tid < n) {
    const int c = rank * BJ_W + tid;
    lam32[c] = __ldcg(A + (size_t)c * ne + c);
  }
}

// Ranks of the FP32 eigenvalues (every block forms them): pos[i] = place of i among the kk
// largest or -1, lead[j] = index of the j-th; the blocks gather the leading vectors into Xk
// (kk x n).  state: [0] the Frobenius norm of A, [1..] the largest correction of iteration
// 0, 1, ... (as float bits).
__global__ void __launch_bounds__(LE_MAXN)
    k_lead_init(int n, const int* __restrict__ nref, const float* __restrict__ lam32, const double* __restrict__ X,
                int* __restrict__ pos, int* __restrict__ lead, double* __restrict__ Xk,
                float* __restrict__ state) {
  __shared__ float lam[LE_MAXN];
  __shared__ int key[LE_MAXN], ld[LE_MAXN];
  __shared__ float red[LE_MAXN / 32];
  const int i = threadIdx.x, kk = *nref;
  if (i < n) {
    lam[i] = lam32[i];
    key[i] = eig_key(lam[i]);
  }
  __syncthreads();
  if (i < n) {
    const int ki = key[i];
    int rank = 0;
    for (int j = 0; j < n; ++j) rank += eig_before(key[j], j, ki, i);
    if (rank < kk) ld[rank] = i;
    if (blockIdx.x == 0) {
      pos[i] = rank < kk ? rank : -1;
      if (rank < kk) lead[rank] = i;
    }
  }
  __syncthreads();
  for (int e = blockIdx.x * LE_MAXN + i; e < kk * n; e += gridDim.x * LE_MAXN)
    Xk[e] = X[(size_t)(e % n) * n + ld[e / n]];
  if (blockIdx.x == 0) {
    float s = i < n ? lam[i] * lam[i] : 0.f;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((i & 31) == 0) red[i >> 5] = s;
    __syncthreads();
    if (i == 0) {
      float t = 0.f;
      for (int w = 0; w < LE_MAXN / 32; ++w) t += red[w];
      state[0] = sqrtf(t);
      for (int it = 1; it <= LE_ITERS; ++it) state[it] = 0.f;
    }
  }
}

// An iteration has nothing left to do once the previous one's largest correction was below
// 1e-13: its own would be the basis error (at most 1e-3 of a gap) times that.
__device__ __forceinline__ bool lead_done(const float* state, int it) {
  return it > 0 && state[it] <= 1e-13f;
}

// U = A Xk' by one warp per (row i, vector j); the refined vectors take their columns in X.
__global__ void __launch_bounds__(256)
    k_lead_u(int n, const int* __restrict__ nref, int it, const double* __restrict__ A, const double* __restrict__ Xk,
             const int* __restrict__ lead, const float* __restrict__ state,
             double* __restrict__ U, double* __restrict__ X) {
  if (lead_done(state, it)) return;
  const int w = (int)((blockIdx.x * 256u + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (w >= n * *nref) return;
  const int j = w / n, i = w - j * n;
  double s = 0.0;
  for (int m = lane; m < n; m += 32) s = fma(A[(size_t)i * n + m], Xk[(size_t)j * n + m], s);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) {
    U[(size_t)j * n + i] = s;
    X[(size_t)i * n + lead[j]] = Xk[(size_t)j * n + i];
  }
}

// S[j][i] = X_i' U_j and R[j][i] = delta - X_i' Xk_j: block (32 columns i, vector j), 32
// warps over the rows m (short FP64 chains), their sums added in shared memory.
__global__ void __launch_bounds__(1024)
    k_lead_sr(int n, const int* __restrict__ nref, int it, const double* __restrict__ X, const double* __restrict__ Xk,
              const double* __restrict__ U, const int* __restrict__ pos,
              const float* __restrict__ state, double* __restrict__ S, double* __restrict__ R) {
  __shared__ double ps[32][33], pr[32][33];
  if (lead_done(state, it) || (int)blockIdx.y >= *nref) return;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane, j = blockIdx.y;
  double s = 0.0, r = 0.0;
  if (i < n)
    for (int m = wp; m < n; m += 32) {
      const double x = X[(size_t)m * n + i];
      s = fma(x, U[(size_t)j * n + m], s);
      r = fma(x, Xk[(size_t)j * n + m], r);
    }
  ps[wp][lane] = s;
  pr[wp][lane] = r;
  __syncthreads();
  // warp wp adds column wp of both
  s = ps[lane][wp];
  r = pr[lane][wp];
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  const int c = blockIdx.x * 32 + wp;
  if (lane == 0 && c < n) {
    S[(size_t)j * n + c] = s;
    R[(size_t)j * n + c] = (pos[c] == j ? 1.0 : 0.0) - r;
  }
}

// Corrections e_i of vector j (blockIdx.x; each of its blocks forms them all, which takes less
// than a launch of their own), then Xk_j += X e on the rows of blockIdx.y, a warp a row.
// Pairs closer than 2 (|off-diagonal S_j| + |A| |R_j|) are a cluster: only made orthogonal (by
// both vectors where both are refined, else by x_j alone).  state[1 + it] takes the largest
// correction of the k wanted vectors, 1 while a cluster still couples by more than 1e-13 |A|.
constexpr int LX_BLOCKS = 8;  // row blocks of a vector
__global__ void __launch_bounds__(LE_MAXN)
    k_lead_ex(int n, int k, const int* __restrict__ nref, int it, const float* __restrict__ lam32,
              const int* __restrict__ pos, const int* __restrict__ lead,
              const double* __restrict__ S, const double* __restrict__ R,
              const double* __restrict__ X, double* __restrict__ Xk, double* __restrict__ lamk,
              float* __restrict__ state) {
  __shared__ float red[LE_MAXN / 32][2];
  __shared__ double es[LE_MAXN];
  if (lead_done(state, it) || (int)blockIdx.x >= *nref) return;
  const int i = threadIdx.x, j = blockIdx.x, self = lead[j];
  const bool in = i < n;
  const double s = in ? S[(size_t)j * n + i] : 0.0, r = in ? R[(size_t)j * n + i] : 0.0;
  const float sf = i == self ? 0.f : (float)s, rf = (float)r;
  float so = sf * sf, rn = rf * rf;
  for (int o = 16; o > 0; o >>= 1) {
    so += __shfl_xor_sync(0xffffffffu, so, o);
    rn += __shfl_xor_sync(0xffffffffu, rn, o);
  }
  if ((i & 31) == 0) {
    red[i >> 5][0] = so;
    red[i >> 5][1] = rn;
  }
  __syncthreads();
  so = rn = 0.f;
  for (int w = 0; w < LE_MAXN / 32; ++w) {
    so += red[w][0];
    rn += red[w][1];
  }
  const float delta = 2.f * (sqrtf(so) + state[0] * sqrtf(rn));
  auto ritz = [&](int v) {  // refined eigenvalue of leading vector v
    return S[(size_t)v * n + lead[v]] / (1.0 - R[(size_t)v * n + lead[v]]);
  };
  const double lj = ritz(j);
  float mag = 0.f;
  if (in) {
    const double li = pos[i] >= 0 ? ritz(pos[i]) : (double)lam32[i];
    const double gap = lj - li;
    const double couple = s + lj * r;
    const bool close = fabs(gap) <= (double)delta;
    const double e = i == self ? 0.5 * r : close ? (pos[i] >= 0 ? 0.5 * r : r) : couple / gap;
    es[i] = e;
    mag = fabsf((float)e);
    if (close && i != self && fabs(couple) > 1e-13 * (double)state[0]) mag = 1.f;
  }
  if (blockIdx.y == 0) {
    for (int o = 16; o > 0; o >>= 1) mag = fmaxf(mag, __shfl_xor_sync(0xffffffffu, mag, o));
    // (a NaN compares as larger than any number here: not converged)
    if ((i & 31) == 0 && j < k)
      atomicMax(reinterpret_cast<int*>(state + 1 + it), __float_as_int(mag) & 0x7fffffff);
    if (i == 0) lamk[j] = lj;
  }
  __syncthreads();
  const int lane = i & 31;
  for (int m = blockIdx.y * (LE_MAXN / 32) + (i >> 5); m < n; m += LX_BLOCKS * (LE_MAXN / 32)) {
    double a = 0.0;
    for (int c = lane; c < n; c += 32) a = fma(X[(size_t)m * n + c], es[c], a);
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) Xk[(size_t)j * n + m] += a;
  }
}

// The FP64 fall-back's first half, when the last iteration over the leading vectors left a
// correction above LE_BAD: X0 (the untouched FP32 basis) made orthonormal by two
// Newton-Schulz steps X <- X + X (I - X'X) / 2 (1e-6 -> 1e-12 -> 1e-24), then S = X'AX.
// One cooperative launch, so that a matrix that does not need it pays one empty launch.
constexpr float LE_BAD = 1e-10f;
__global__ void __launch_bounds__(LE_MAXN)
    k_lead_full(int n, const float* __restrict__ state, const double* __restrict__ A,
                double* __restrict__ X, double* __restrict__ U, double* __restrict__ S) {
  if (!(state[LE_ITERS] > LE_BAD)) return;  // the same value in every block
  const cg::grid_group grid = cg::this_grid();
  __shared__ double row[LE_MAXN];
  const int t = threadIdx.x;
  // row i of op(L) M, column t, two chains
  auto rowmm = [&](const double* L, bool tl, const double* M, int i) {
    __syncthreads();
    if (t < n) row[t] = tl ? __ldcg(L + (size_t)t * n + i) : __ldcg(L + (size_t)i * n + t);
    __syncthreads();
    double s0 = 0.0, s1 = 0.0;
    if (t < n) {
      int k = 0;
      for (; k + 1 < n; k += 2) {
        s0 = fma(row[k], __ldcg(M + (size_t)k * n + t), s0);
        s1 = fma(row[k + 1], __ldcg(M + (size_t)(k + 1) * n + t), s1);
      }
      if (k < n) s0 = fma(row[k], __ldcg(M + (size_t)k * n + t), s0);
    }
    return s0 + s1;
  };
  for (int step = 0; step < 2; ++step) {
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
      const double xx = rowmm(X, true, X, i);
      if (t < n) U[(size_t)i * n + t] = (i == t ? 1.0 : 0.0) - xx;
    }
    grid.sync();
    for (int i = blockIdx.x; i < n; i += gridDim.x) {  // a row is read whole before it is written
      const double x = rowmm(X, false, U, i);
      if (t < n) X[(size_t)i * n + t] = fma(0.5, x, row[t]);
    }
    grid.sync();
  }
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    const double ax = rowmm(A, false, X, i);
    if (t < n) U[(size_t)i * n + t] = ax;
  }
  grid.sync();
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    const double s = rowmm(X, true, U, i);
    if (t < n) S[(size_t)i * n + t] = s;
  }
}

// Cyclic Jacobi in FP64 on Ma = X'AX (symmetrised here, nearly diagonal), the rotations
// applied to the columns of X, lam <- its diagonal: round-robin rounds of n / 2 disjoint
// rotations, of each sweep only those rounds that hold an entry above 1e-14 |A|.  One
// cooperative launch, gated like the steps that make X'AX.  n <= 1024.
constexpr int CR_SWEEPS = 12;
constexpr int CR_MAXN = 1024;
__global__ void __launch_bounds__(256)
    k_rotate(int n, const float* __restrict__ gate, float limit, const double* __restrict__ S,
             double* __restrict__ lam, double* __restrict__ X, double* __restrict__ Ma,
             double* __restrict__ Mb, double* __restrict__ normsq, int* __restrict__ flag) {
  if (!(*gate > limit)) return;  // the same value in every block
  const cg::grid_group grid = cg::this_grid();
  __shared__ double cs[CR_MAXN];  // (c, s) of each pair
  __shared__ double red[8];
  const int ne = (n + 1) & ~1, np = ne / 2, t = threadIdx.x;
  int* any = flag + ne;  // one per sweep
  if (blockIdx.x == 0) {
    if (t < CR_SWEEPS) any[t] = 0;
    if (t == 0) *normsq = 0.0;
  }
  grid.sync();
  double sq = 0.0;
  for (int p = blockIdx.x; p < n; p += gridDim.x)
    for (int q = t; q < n; q += 256) {
      const double m = 0.5 * (S[(size_t)p * n + q] + S[(size_t)q * n + p]);
      Ma[(size_t)p * n + q] = m;
      sq += m * m;
    }
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  if ((t & 31) == 0) red[t >> 5] = sq;
  __syncthreads();
  if (t == 0) {
    for (int w = 1; w < 8; ++w) sq += red[w];
    atomicAdd(normsq, sq);
  }
  grid.sync();
  const double tol = 1e-14 * sqrt(__ldcg(normsq));
  for (int sweep = 0; sweep < CR_SWEEPS; ++sweep) {
    for (int r = blockIdx.x; r < ne - 1; r += gridDim.x) {
      int hit = 0;
      for (int i = t; i < np; i += 256) {
        int p, q;
        rr_pair(ne, r, i, p, q);
        hit |= q < n && fabs(__ldcg(Ma + (size_t)p * n + q)) > tol;
      }
      hit = __syncthreads_or(hit);
      if (t == 0) {
        flag[r] = hit;
        if (hit) atomicOr(any + sweep, 1);
      }
    }
    grid.sync();
    if (__ldcg(any + sweep) == 0) break;
    for (int r = 0; r < ne - 1; ++r) {
      if (__ldcg(flag + r) == 0) continue;
      __syncthreads();
      for (int i = t; i < np; i += 256) {
        int p, q;
        rr_pair(ne, r, i, p, q);
        double c = 1.0, sn = 0.0;
        const double a = q < n ? __ldcg(Ma + (size_t)p * n + q) : 0.0;
        if (fabs(a) > tol) {
          const double tau =
              (__ldcg(Ma + (size_t)q * n + q) - __ldcg(Ma + (size_t)p * n + p)) / (2.0 * a);
          const double tt = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
          c = 1.0 / sqrt(1.0 + tt * tt);
          sn = tt * c;
        }
        cs[2 * i] = c;
        cs[2 * i + 1] = sn;
      }
      __syncthreads();
      for (int bi = blockIdx.x; bi < np; bi += gridDim.x) {
        int pi, qi;
        rr_pair(ne, r, bi, pi, qi);
        const double ci = cs[2 * bi], si = cs[2 * bi + 1];
        const bool vi = qi < n;
        for (int bj = t; bj < np; bj += 256) {
          int pj, qj;
          rr_pair(ne, r, bj, pj, qj);
          const double cj = cs[2 * bj], sj = cs[2 * bj + 1];
          const bool vj = qj < n;
          const double m00 = __ldcg(Ma + (size_t)pi * n + pj);
          const double m01 = vj ? __ldcg(Ma + (size_t)pi * n + qj) : 0.0;
          const double m10 = vi ? __ldcg(Ma + (size_t)qi * n + pj) : 0.0;
          const double m11 = vi && vj ? __ldcg(Ma + (size_t)qi * n + qj) : 0.0;
          const double c00 = cj * m00 - sj * m01, c01 = sj * m00 + cj * m01;
          const double c10 = cj * m10 - sj * m11, c11 = sj * m10 + cj * m11;
          Mb[(size_t)pi * n + pj] = ci * c00 - si * c10;
          if (vj) Mb[(size_t)pi * n + qj] = ci * c01 - si * c11;
          if (vi) Mb[(size_t)qi * n + pj] = si * c00 + ci * c10;
          if (vi && vj) Mb[(size_t)qi * n + qj] = si * c01 + ci * c11;
        }
      }
      for (int m = blockIdx.x; m < n; m += gridDim.x)  // a block owns its rows of X
        for (int i = t; i < np; i += 256) {
          int p, q;
          rr_pair(ne, r, i, p, q);
          const double c = cs[2 * i], sn = cs[2 * i + 1];
          if (q >= n || sn == 0.0) continue;
          const double xp = X[(size_t)m * n + p], xq = X[(size_t)m * n + q];
          X[(size_t)m * n + p] = c * xp - sn * xq;
          X[(size_t)m * n + q] = sn * xp + c * xq;
        }
      grid.sync();
      double* sw = Ma;
      Ma = Mb;
      Mb = sw;
    }
    grid.sync();  // every block is past this sweep's flags before the next sweep writes them
  }
  for (int p = blockIdx.x * 256 + t; p < n; p += gridDim.x * 256)
    lam[p] = __ldcg(Ma + (size_t)p * n + p);
}

// The k largest eigenvalues in descending order (ties by place) and their vectors: of the kk
// refined ones (blocks 0..kk-1), or of all n (columns of X) after the fall-back.
__global__ void __launch_bounds__(LE_MAXN)
    k_lead_out(int n, const int* __restrict__ nref, int k, const float* __restrict__ state,
               const double* __restrict__ lamk, const double* __restrict__ Xk,
               const double* __restrict__ lam, const double* __restrict__ X,
               double* __restrict__ theta, double* __restrict__ psi, int* __restrict__ order) {
  const bool full = state[LE_ITERS] > LE_BAD;
  const int j = blockIdx.x, t = threadIdx.x, nv = full ? n : *nref;
  if (j >= nv) return;
  const double* l = full ? lam : lamk;
  const double lj = l[j];
  const int rank = __syncthreads_count(t < nv && eig_before(eig_key(l[t]), t, eig_key(lj), j));
  if (rank >= k) return;
  if (t < n) psi[(size_t)rank * n + t] = full ? X[(size_t)t * n + j] : Xk[(size_t)j * n + t];
  if (t == 0) {
    theta[rank] = lj;
    order[rank] = rank;
  }
}

}  // namespace

// One cluster holds the whole matrix up to n = 256.  Beyond, the launches of
// launch_dense_eig spread a round's products over more SMs than a cluster has.
bool lead_eig_takes(int n) { return n <= LE_MAXN; }

int rotate_ints(int n) { return n + 2 + CR_SWEEPS; }

fpca_status launch_rotate(fpca_ctx* ctx, int n, const float* gate, float limit, const double* S,
                          double* lam, double* X, double* Ma, double* Mb, double* normsq,
                          int* flag) {
  void* args[] = {(void*)&n, (void*)&gate, (void*)&limit, (void*)&S, &lam, &X, &Ma, &Mb, &normsq,
                  &flag};
  // one block per SM at most: all resident, as the grid barrier needs
  cudaLaunchCooperativeKernel((const void*)k_rotate, dim3(std::min(n, ctx->num_sms)), dim3(256),
                              args, 0, ctx->stream);
  FPCA_LAUNCHED(ctx, "eig_rotate");
  return FPCA_OK;
}

size_t lead_eig_bytes(int n, int k) {
  const size_t ne = le_ne(n), kk = std::min(n, k + LE_EXTRA);
  return WsCarve::round(sizeof(float) * ne * ne) + WsCarve::round(sizeof(double) * (size_t)n * n) +
         WsCarve::round(sizeof(float) * n) + 2 * WsCarve::round(sizeof(int) * n) + WsCarve::round(sizeof(int)) +
         WsCarve::round(sizeof(float) * (LE_ITERS + 1)) +
         4 * WsCarve::round(sizeof(double) * kk * n) + WsCarve::round(sizeof(double) * kk) +
         4 * WsCarve::round(sizeof(double) * (size_t)n * n) + WsCarve::round(sizeof(double) * n) +
         WsCarve::round(sizeof(double)) + WsCarve::round(sizeof(int) * rotate_ints(n)) + 4096;
}

fpca_status launch_lead_eig(fpca_ctx* ctx, int n, int k, const double* S, double* theta,
                            double* psi, int* order, void* scratch) {
  const int ne = le_ne(n), kk = std::min(n, k + LE_EXTRA);
  WsCarve c(scratch);
  float* Af = c.take<float>((size_t)ne * ne);
  double* X = c.take<double>((size_t)n * n);
  float* lam32 = c.take<float>(n);
  int* pos = c.take<int>(n);
  int* lead = c.take<int>(n);
  int* nref = c.take<int>(1);
  float* state = c.take<float>(LE_ITERS + 1);
  double* Xk = c.take<double>((size_t)kk * n);
  double* U = c.take<double>((size_t)kk * n);
  double* Sx = c.take<double>((size_t)kk * n);
  double* R = c.take<double>((size_t)kk * n);
  double* lamk = c.take<double>(kk);
  double* X0 = c.take<double>((size_t)n * n);
  double* Uf = c.take<double>((size_t)n * n);
  double* Sf = c.take<double>((size_t)n * n);
  double* Mf = c.take<double>((size_t)n * n);
  double* lamf = c.take<double>(n);
  double* normsq = c.take<double>(1);
  int* flag = c.take<int>(rotate_ints(n));
  const size_t sm = le_smem(ne);
  cudaFuncSetAttribute(k_bj_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ne / BJ_W);
  cfg.blockDim = dim3(BJ_NT);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = ctx->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ne / BJ_W;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_bj_cluster, n, ne, k, kk, S, Af, X, X0, lam32, nref);
  FPCA_LAUNCHED(ctx, "eig_bj_cluster");
  k_lead_init<<<8, LE_MAXN, 0, ctx->stream>>>(n, nref, lam32, X, pos, lead, Xk, state);
  FPCA_LAUNCHED(ctx, "eig_lead_init");
  const int wb = (n * kk + 7) / 8;  // blocks of 8 warps, one warp per (row, vector)
  for (int it = 0; it < LE_ITERS; ++it) {
    k_lead_u<<<wb, 256, 0, ctx->stream>>>(n, nref, it, S, Xk, lead, state, U, X);
    FPCA_LAUNCHED(ctx, "eig_lead_u");
    k_lead_sr<<<dim3((n + 31) / 32, kk), 1024, 0, ctx->stream>>>(n, nref, it, X, Xk, U, pos, state, Sx, R);
    FPCA_LAUNCHED(ctx, "eig_lead_sr");
    k_lead_ex<<<dim3(kk, LX_BLOCKS), LE_MAXN, 0, ctx->stream>>>(n, k, nref, it, lam32, pos, lead, Sx, R,
                                                               X, Xk, lamk, state);
    FPCA_LAUNCHED(ctx, "eig_lead_x");
  }
  {
    const float* st = state;
    void* args[] = {(void*)&n, &st, (void*)&S, &X0, &Uf, &Sf};
    // one block per SM at most: all resident, as the grid barrier needs
    cudaLaunchCooperativeKernel((const void*)k_lead_full, dim3(std::min(n, ctx->num_sms)),
                                dim3(LE_MAXN), args, 0, ctx->stream);
    FPCA_LAUNCHED(ctx, "eig_lead_full");
  }
  fpca_status cs = launch_rotate(ctx, n, state + LE_ITERS, LE_BAD, Sf, lamf, X0, Mf, Uf, normsq, flag);
  if (cs != FPCA_OK) return cs;
  k_lead_out<<<n, LE_MAXN, 0, ctx->stream>>>(n, nref, k, state, lamk, Xk, lamf, X0, theta, psi, order);
  FPCA_LAUNCHED(ctx, "eig_lead_out");
  return FPCA_OK;
}
