// Binning (Section 3.2) of the sums in Eq. (2.3) and Eq. (2.4).
//
// Mean bins carry, per grid bin b: the observation count, W_b = sum 1/N_i and
// V_b = sum Y_ij / N_i (V2 with Y^2).  Covariance bins carry, per ordered
// bin pair (p, q): the pair count, W = sum w_i, V = sum w_i R_ij R_il with
// w_i = 1/(N_i (N_i - 1)), over pairs j != l of one subject.
#include <algorithm>

#include <cuda_bf16.h>

#include "fpca_internal.cuh"
#include "ff.cuh"

namespace {

__device__ __forceinline__ double load_y(const void* y, int prec, size_t idx) {
  return prec == FPCA_F64 ? static_cast<const double*>(y)[idx]
                          : static_cast<double>(static_cast<const float*>(y)[idx]);
}

__device__ __forceinline__ int bin_index(const double* t, int d, const int* m) {
  int flat = 0;
  for (int k = 0; k < d; ++k) {
    double x = floor(__dmul_rn(t[k], (double)m[k]));
    int ik = (int)fmin(fmax(x, 0.0), (double)(m[k] - 1));
    flat = flat * m[k] + ik;
  }
  return flat;
}

// N_i: observed nodes of subject i (mask row sum), one warp per subject; rows
// are read 16 bytes at a time when they are 16-byte aligned.
__global__ void k_subject_counts(int n, int P, const uint8_t* __restrict__ mask,
                                 int32_t* __restrict__ Ni) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= n) return;
  int c = 0;
  if (!mask) {
    c = lane == 0 ? P : 0;
  } else if (P % 16 == 0 && (reinterpret_cast<uintptr_t>(mask) & 15) == 0) {
    const uint4* row = reinterpret_cast<const uint4*>(mask + (size_t)i * P);
    for (int q = lane; q < P / 16; q += 32) {
      const uint4 v = row[q];
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)  // count the nonzero bytes of w[k]
        c += __popc(__vcmpne4(w[k], 0u)) >> 3;
    }
  } else {
    const uint8_t* row = mask + (size_t)i * P;
    for (int p = lane; p < P; p += 32) c += row[p] != 0;
  }
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) Ni[i] = c;
}

// Dense mean bins: a block covers 32 nodes; its MB_SLICES thread rows take
// every MB_SLICES-th subject, and the partial sums are added by a fixed
// pairwise tree (deterministic).  Weights 1/N_i.
constexpr int MB_SLICES = 32;  // subject slices per block: short FP64 add chains
constexpr int MB_BATCH = 8;    // subjects whose loads are issued together (4 for FP64 y)
template <typename TY>
__global__ void __launch_bounds__(32 * MB_SLICES)
    k_bin_mean_dense(int n, int P, const TY* __restrict__ y, const uint8_t* __restrict__ mask,
                     const int32_t* __restrict__ Ni, int32_t* __restrict__ cnt,
                     double* __restrict__ w, double* __restrict__ v, double* __restrict__ v2) {
  __shared__ double ps[3][MB_SLICES][32];
  __shared__ int pc[MB_SLICES][32];
  __shared__ float winvh[32 * MB_SLICES], winvl[32 * MB_SLICES];
  const int p = blockIdx.x * 32 + threadIdx.x;
  int c = 0;
  // per-thread sums in float-float (about 48 bits from FP32 operations: FP64
  // adds are long-latency and low-throughput on this GPU), joined in FP64 below
  ff::F2 fw = ff::make(0.f), fv = ff::make(0.f), fv2 = ff::make(0.f);
  const int tid = threadIdx.y * 32 + threadIdx.x;
  for (int i0 = 0; i0 < n; i0 += 32 * MB_SLICES) {
    // 1/N_i for the next 32 * MB_SLICES subjects, one division per subject
    __syncthreads();
    {
      const int i = i0 + tid;
      const int N = i < n ? Ni[i] : 0;
      const double wd = N > 0 ? 1.0 / (double)N : 0.0;
      const float hi = (float)wd;
      winvh[tid] = hi;
      winvl[tid] = (float)(wd - (double)hi);
    }
    __syncthreads();
    if (p < P) {
      const int iend = min(n, i0 + 32 * MB_SLICES);
      constexpr int NB = sizeof(TY) == 8 ? MB_BATCH / 2 : MB_BATCH;
      for (int ib = i0 + threadIdx.y; ib < iend; ib += NB * MB_SLICES) {
        // the batch's loads first (independent of the sums), then the sums in
        // subject order
        TY yb[NB];
        bool ok[NB];
#pragma unroll
        for (int u = 0; u < NB; ++u) {
          const int i = ib + u * MB_SLICES;
          const size_t idx = (size_t)i * P + p;
          ok[u] = i < iend && (!mask || mask[idx]);
          yb[u] = i < iend ? y[idx] : TY(0);
        }
#pragma unroll
        for (int u = 0; u < NB; ++u) {
          const int i = ib + u * MB_SLICES;
          if (!ok[u]) continue;
          const ff::F2 wi = {winvh[i - i0], winvl[i - i0]};
          if (wi.hi == 0.f) continue;
          ff::F2 yy, y2;
          if constexpr (sizeof(TY) == 8) {
            const double yd = yb[u];
            const float hi = (float)yd;
            yy = {hi, (float)(yd - (double)hi)};
            y2 = ff::mul(yy, yy);
          } else {
            const float yf = yb[u];
            yy = ff::make(yf);
            y2 = ff::two_prod(yf, yf);  // exact
          }
          c += 1;
          fw = ff::add(fw, wi);
          fv = ff::add(fv, ff::mul(wi, yy));
          fv2 = ff::add(fv2, ff::mul(wi, y2));
        }
      }
    }
  }
  const double sw = ff::to_double(fw), sv = ff::to_double(fv), sv2 = ff::to_double(fv2);
  ps[0][threadIdx.y][threadIdx.x] = sw;
  ps[1][threadIdx.y][threadIdx.x] = sv;
  ps[2][threadIdx.y][threadIdx.x] = sv2;
  pc[threadIdx.y][threadIdx.x] = c;
  __syncthreads();
  // pairwise tree over the slices (fixed order; FP64 adds have a long latency)
  for (int h = MB_SLICES / 2; h >= 1; h >>= 1) {
    if (threadIdx.y < h) {
      pc[threadIdx.y][threadIdx.x] += pc[threadIdx.y + h][threadIdx.x];
#pragma unroll
      for (int a = 0; a < 3; ++a) ps[a][threadIdx.y][threadIdx.x] += ps[a][threadIdx.y + h][threadIdx.x];
    }
    __syncthreads();
  }
  if (threadIdx.y == 0 && p < P) {
    cnt[p] = pc[0][threadIdx.x];
    w[p] = ps[0][0][threadIdx.x];
    v[p] = ps[1][0][threadIdx.x];
    if (v2) v2[p] = ps[2][0][threadIdx.x];
  }
}

// Sparse mean bins: one thread per subject, atomic scatter into the bins.
__global__ void k_bin_mean_sparse(int n, long long N, int d, int m0, int m1, int m2,
                                  const int64_t* __restrict__ offs, const double* __restrict__ t,
                                  const double* __restrict__ y, int32_t* cnt, double* w,
                                  double* v, double* v2, int* __restrict__ err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int m[3] = {m0, m1, m2};
  const int64_t lo = offs[i], hi = offs[i + 1];
  if (lo < 0 || hi < lo || hi > N) {
    atomicExch(err, DERR_BOUNDS);
    return;
  }
  if (hi == lo) return;
  const double wi = 1.0 / (double)(hi - lo);
  for (int64_t j = lo; j < hi; ++j) {
    const int b = bin_index(t + j * d, d, m);
    const double yy = y[j];
    atomicAdd(cnt + b, 1);
    atomicAdd(w + b, wi);
    atomicAdd(v + b, __dmul_rn(wi, yy));
    if (v2) atomicAdd(v2 + b, __dmul_rn(wi, __dmul_rn(yy, yy)));
  }
}

// Operand planes of the tensor-core Gram products, K-major (subject index
// contiguous), BF16, zero-padded to Kpad subjects:
//   plane 0: M_ip                 (pair counts  C = M'M)
//   plane 1: w_i M_ip             (W = (wM)'M, exact 0/1 right operand)
//   plane 2: sqrt(w_i) R_ip M_ip  (V = R~'R~)
// A tile of 64 subjects x 32 nodes is transposed through shared memory: the
// reads run along the nodes (y, mask), the writes along the subjects as BF16
// pairs (128 bytes per node and plane).
template <typename TY>
__global__ void __launch_bounds__(256)
    k_cov_operands_bf16(int n, int P, int Kpad, const TY* __restrict__ y,
                        const uint8_t* __restrict__ mask, const int32_t* __restrict__ Ni,
                        const double* __restrict__ mu, int mode, __nv_bfloat162* __restrict__ ops) {
  __shared__ float tw[64][33], tr[64][33];
  __shared__ uint8_t tm[64][36];
  __shared__ float wsub[64], swsub[64], muf[32];
  const int i0 = blockIdx.y * 64, p0 = blockIdx.x * 32;
  const int tid = threadIdx.y * 32 + threadIdx.x;
  // per-subject weights w_i = 1/(N_i (N_i - 1)) and sqrt(w_i), and the mean at the
  // block's 32 nodes, once per block and in FP32: the operands are rounded to
  // BF16, so FP32 is ample (and FP64 operations are slow on this GPU)
  if (tid < 64) {
    const int i = i0 + tid;
    const int N = i < n ? Ni[i] : 0;
    const float wi = N >= 2 ? 1.f / ((float)N * (float)(N - 1)) : 0.f;
    wsub[tid] = wi;
    swsub[tid] = sqrtf(wi);
  } else if (tid < 96) {
    const int p = p0 + tid - 64;
    muf[tid - 64] = (p < P && mode == FPCA_COV_RESIDUAL) ? (float)mu[p] : 0.f;
  }
  // this thread's 8 observations, loads first (mask and y together)
  TY yv[8];
  uint8_t ob[8];
  const int p = p0 + threadIdx.x;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int i = i0 + threadIdx.y + 8 * u;
    const bool in = i < n && p < P;
    const size_t idx = (size_t)i * P + p;
    ob[u] = in ? (mask ? mask[idx] : (uint8_t)1) : (uint8_t)0;
    yv[u] = in ? y[idx] : TY(0);
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int r = threadIdx.y + 8 * u;
    const bool obs = ob[u] != 0;
    tm[r][threadIdx.x] = obs ? 1 : 0;
    tw[r][threadIdx.x] = obs ? wsub[r] : 0.f;
    tr[r][threadIdx.x] = obs ? swsub[r] * ((float)yv[u] - muf[threadIdx.x]) : 0.f;
  }
  __syncthreads();
  // node p0 + c, subjects i0 + 2 lane and i0 + 2 lane + 1
  const size_t plane = (size_t)P * Kpad / 2;   // in BF16 pairs
  for (int c = threadIdx.y; c < 32; c += 8) {
    const int pn = p0 + c;
    if (pn >= P) continue;
    const int a = 2 * threadIdx.x;
    const size_t o = ((size_t)pn * Kpad + i0) / 2 + threadIdx.x;
    ops[o] = __floats2bfloat162_rn((float)tm[a][c], (float)tm[a + 1][c]);
    ops[plane + o] = __floats2bfloat162_rn(tw[a][c], tw[a + 1][c]);
    ops[2 * plane + o] = __floats2bfloat162_rn(tr[a][c], tr[a + 1][c]);
  }
}

// FP64 covariance bins of gridded data: an 8 x 8 output tile a block, tiles on and above the
// diagonal (the ones below are their transposes), subjects streamed through shared memory.
// FP64 runs at two results a clock on an SM here, so the tiles are small enough to give every
// SM some at 64 nodes, and a pair costs three FP64 operations: the weight enters a subject's
// row once, and the pair's weight is selected, not multiplied.  16 x 16 tiles of the whole
// matrix with six operations took 65 us at 64 nodes, n = 100, and 60 us at 256, n = 50; these
// take 26 and 20.
constexpr int CD_T = 8;     // tile edge
constexpr int CD_K = 32;    // subjects at a time
constexpr int CD_W = 256;   // subjects whose weights are formed at a time
__global__ void __launch_bounds__(CD_T * CD_T)
    k_cov_dense_f64(int n, int P, int nt, const void* __restrict__ y, int y_prec,
                    const uint8_t* __restrict__ mask, const int32_t* __restrict__ Ni,
                    const double* __restrict__ mu, int mode, int32_t* __restrict__ cnt,
                    double* __restrict__ w, double* __restrict__ v) {
  __shared__ double rp[CD_K][CD_T + 1], rq[CD_K][CD_T + 1], wsub[CD_W];
  __shared__ uint8_t mp[CD_K][CD_T], mq[CD_K][CD_T];
  // tile pair (bi <= bj): bj runs fastest
  int bi = 0, bj = (int)blockIdx.x;
  while (bj >= nt - bi) bj -= nt - bi++;
  bj += bi;
  const int tid = threadIdx.x, tx = tid % CD_T, ty = tid / CD_T;
  int c = 0;
  double sw = 0.0, sv = 0.0;
  for (int i0 = 0; i0 < n; i0 += CD_K) {
    if (i0 % CD_W == 0) {
      for (int e = tid; e < CD_W && i0 + e < n; e += CD_T * CD_T) {
        const double N = (double)Ni[i0 + e];
        wsub[e] = N >= 2.0 ? 1.0 / (N * (N - 1.0)) : 0.0;
      }
      __syncthreads();
    }
    const int kmax = min(CD_K, n - i0);
    const double* wc = wsub + i0 % CD_W;
#pragma unroll
    for (int u = 0; u < 2 * CD_K / CD_T; ++u) {  // both sides, CD_T subjects at a time
      const bool rows = u < CD_K / CD_T;
      const int k = (u % (CD_K / CD_T)) * CD_T + ty, at = (rows ? bi : bj) * CD_T + tx;
      bool ob = false;
      double r = 0.0;
      if (k < kmax && at < P) {
        const size_t idx = (size_t)(i0 + k) * P + at;
        ob = !mask || mask[idx] != 0;
        if (ob) {
          const double yy = load_y(y, y_prec, idx);
          r = mode == FPCA_COV_RESIDUAL ? yy - mu[at] : yy;
        }
      }
      if (rows) {
        mp[k][tx] = ob;
        rp[k][tx] = k < kmax ? wc[k] * r : 0.0;
      } else {
        mq[k][tx] = ob;
        rq[k][tx] = r;
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < kmax; ++k) {
      const bool both = mp[k][ty] & mq[k][tx];
      c += both;
      sw = __dadd_rn(sw, both ? wc[k] : 0.0);
      sv = __dadd_rn(sv, __dmul_rn(rp[k][ty], rq[k][tx]));
    }
    __syncthreads();
  }
  const int p = bi * CD_T + ty, q = bj * CD_T + tx;
  if (p < P && q < P) {
    if (p == q) {  // only pairs of an observation with itself
      c = 0;
      sw = sv = 0.0;
    }
    const size_t o = (size_t)p * P + q, ot = (size_t)q * P + p;
    cnt[o] = c;
    w[o] = sw;
    v[o] = sv;
    if (bi != bj) {
      cnt[ot] = c;
      w[ot] = sw;
      v[ot] = sv;
    }
  }
}

// ---------------------------------------------------------------------------
// Covariance bins of scattered data, row by row.  The observations are grouped by
// (fold, bin): one row of the output arrays holds exactly the pairs whose first
// observation lies in that bin, so a CTA sums a row in shared memory and writes every
// entry once.  Rows of more than `chunk` observations are cut into chunks, a CTA each, which
// add their sums to the cleared row.
// ---------------------------------------------------------------------------
struct ObsRec {
  double r;        // response (residual or raw)
  int32_t lo, ni;  // first observation and observation count of its subject
};
// Chunk of a long row: its row and place there (1, 2, ...; a row's first chunk is not listed).
struct RowChunk {
  int32_t row, place;
};

constexpr int OBS_LANES = 8;  // threads per subject

// Per observation: its bin, its record, its weight and its row + 1 (row = fold * P + bin; 0 where
// the subject has no pairs or is skipped).  Offsets outside 0 <= offs[i] <= offs[i+1] <= N and folds
// outside 0..nfold-1 are reported (DERR_BOUNDS) and the subject is skipped.  The caller
// clears row.
// A skipped subject's neighbours can overlap (offsets 0, 10, 5, 12: the first and the third
// both hold observations 5..9).  An observation goes to the subject that claims its row first,
// and only that one writes the record, so that its lo and ni are one checked subject's; it is
// counted and listed by its row, once.  With `rank` the rows are counted here, each observation
// taking its rank in its row; else by k_row_count.
__global__ void k_obs_rows(int n, long long N, int d, int m0, int m1, int m2, int P,
                           const int64_t* __restrict__ offs, const double* __restrict__ t,
                           const double* __restrict__ y, const double* __restrict__ mu, int mode,
                           const int32_t* __restrict__ fold, int nfold, int32_t* __restrict__ ob,
                           ObsRec* __restrict__ rec, double* __restrict__ wt,
                           int32_t* __restrict__ row, int32_t* __restrict__ rowcount,
                           int32_t* __restrict__ rank, int* __restrict__ err) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int i = (int)(g / OBS_LANES), part = (int)(g % OBS_LANES);
  if (i >= n) return;
  const int64_t lo = offs[i], hi = offs[i + 1];
  if (lo < 0 || hi < lo || hi > N) {
    if (part == 0) atomicExch(err, DERR_BOUNDS);
    return;
  }
  if (hi - lo < 2) return;
  int f = 0;
  if (nfold > 0) {
    f = fold[i];
    if (f < 0 || f >= nfold) {
      if (part == 0) atomicExch(err, DERR_BOUNDS);
      return;
    }
  }
  const int m[3] = {m0, m1, m2};
  const double wi = 1.0 / ((double)(hi - lo) * (double)(hi - lo - 1));
  for (int64_t j = lo + part; j < hi; j += OBS_LANES) {
    const int b = bin_index(t + j * d, d, m);
    if (atomicCAS(row + j, 0, f * P + b + 1) != 0) continue;  // another subject's (see above)
    ob[j] = b;
    rec[j] = ObsRec{mode == FPCA_COV_RESIDUAL ? y[j] - mu[b] : y[j], (int32_t)lo,
                    (int32_t)(hi - lo)};
    wt[j] = wi;
    if (rank) rank[j] = atomicAdd(rowcount + f * P + b, 1);
  }
}

// The observation counts of few, long rows and each observation's rank in its row, counted in
// shared memory first: one atomic per block and row, where 250 000 on 64 counters took 60 us.
constexpr int RC_NT = 1024, RC_PER = 4, RC_ROWS = 1024;
__global__ void __launch_bounds__(RC_NT)
    k_row_count(long long N, int rows, const int32_t* __restrict__ row,
                int32_t* __restrict__ rowcount, int32_t* __restrict__ rank) {
  __shared__ int32_t hist[RC_ROWS];
  const long long j0 = blockIdx.x * (long long)(RC_NT * RC_PER) + threadIdx.x;
  int32_t r[RC_PER], k[RC_PER];
#pragma unroll
  for (int u = 0; u < RC_PER; ++u) {
    const long long j = j0 + u * RC_NT;
    r[u] = j < N ? row[j] - 1 : -1;
  }
  for (int e = threadIdx.x; e < rows; e += RC_NT) hist[e] = 0;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < RC_PER; ++u) k[u] = r[u] >= 0 ? atomicAdd(hist + r[u], 1) : 0;
  __syncthreads();
  for (int e = threadIdx.x; e < rows; e += RC_NT)
    if (hist[e] > 0) hist[e] = atomicAdd(rowcount + e, hist[e]);
  __syncthreads();
#pragma unroll
  for (int u = 0; u < RC_PER; ++u)
    if (r[u] >= 0) rank[j0 + u * RC_NT] = hist[r[u]] + k[u];
}

// Each row's place in the list of observations: the rows take consecutive runs in no
// particular order (one atomic per warp), so no scan is needed.  Rows longer than `chunk` list
// their further chunks: at most N / chunk in all.
__global__ void k_row_starts(int rows, int chunk, const int32_t* __restrict__ rowcount,
                             int32_t* __restrict__ start, int32_t* __restrict__ total,
                             int32_t* __restrict__ nextra, RowChunk* __restrict__ extra) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  const int c = r < rows ? rowcount[r] : 0;
  int incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  int base = 0;
  if (lane == 31) base = atomicAdd(total, incl);
  base = __shfl_sync(0xffffffffu, base, 31);
  if (r < rows) start[r] = base + incl - c;
  if (c > chunk) {
    const int more = (c - 1) / chunk, at = atomicAdd(nextra, more);
    for (int k = 0; k < more; ++k) extra[at + k] = RowChunk{r, k + 1};
  }
}

// The lists, and (blocks from `fill` on, one per further chunk) zeros in the rows that are summed
// in chunks; es: bytes of an entry of w, v and q.
__global__ void k_row_fill(long long N, int fill, const int32_t* __restrict__ row,
                           const int32_t* __restrict__ start, const int32_t* __restrict__ rank,
                           int32_t* __restrict__ list, int P, int es,
                           const int32_t* __restrict__ nextra, const RowChunk* __restrict__ extra,
                           int32_t* __restrict__ cnt, void* __restrict__ w, void* __restrict__ v,
                           void* __restrict__ q) {
  if ((int)blockIdx.x >= fill) {
    const int x = blockIdx.x - fill;
    if (x >= *nextra || extra[x].place != 1) return;
    const size_t o = (size_t)extra[x].row * P;
    void* const dst[3] = {w, v, q};
    for (int e = threadIdx.x; e < P; e += blockDim.x) cnt[o + e] = 0;
    for (void* d : dst) {
      if (!d) continue;
      uint32_t* out = reinterpret_cast<uint32_t*>(static_cast<char*>(d) + o * es);
      for (int e = threadIdx.x; e < P * (es / 4); e += blockDim.x) out[e] = 0u;
    }
    return;
  }
  const long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (j >= N) return;
  const int r = row[j] - 1;
  if (r >= 0) list[start[r] + rank[j]] = (int32_t)j;
}

// One chunk of an output row (blockIdx.x < rows: the first chunk of row fold * P + bin, else an
// entry of `extra`), columns [blockIdx.y * PC, + PC): each warp takes up to 32 observations of the
// row at a time (fewer where the chunk would not give every warp some) and its lanes the pairs of
// all of them with the other observations of their subjects; terms as w_i, w_i r r', w_i (r r')^2
// in FP64, rounded to T and added in shared memory.  A row of one chunk goes out by
// one bulk copy per array (or plain stores where a row does not start on 16 bytes); chunks of a
// longer one add what is not zero to the cleared row.
// Large outputs are bound by their write: 20 000 subjects of 5..20 observations on 64 x 64
// bins, 5 folds (1.34 GB, 0.2 ms at 6.8 TB/s) take 0.34 ms for the whole call.  A scatter by global
// atomics took 0.74 ms: it cleared the arrays and added each pair's four terms on lines already
// gone from L2.  Small ones are bound by the FP64 terms (two results a clock and SM), so no lane
// without a pair, and the weight's division once a subject: on 24 x 24 bins 0.28 ms with an
// observation a warp and a division each, 0.11 now (the scatter: 0.12).
// One CTA a row left SMs idle where rows are few, and one SM with a row that holds much of the
// data: 64 bins without folds 0.82 ms, 0.10 now (the scatter: 0.21); half of all observations in
// one bin of 64 x 64 7.5 ms, 0.57 now (the scatter: 1.0).
constexpr int CSR_NT = 256;
constexpr int CSR_CHUNK = 256;   // observations per chunk, at least: 32 a warp
template <typename T>
__global__ void __launch_bounds__(CSR_NT)
    k_cov_rows(int rows, int P, int PC, int chunk, const int32_t* __restrict__ rowcount,
               const int32_t* __restrict__ start, const int32_t* __restrict__ list,
               const int32_t* __restrict__ ob, const ObsRec* __restrict__ rec,
               const double* __restrict__ wt, const int32_t* __restrict__ nextra,
               const RowChunk* __restrict__ extra, int32_t* __restrict__ cnt, T* __restrict__ w,
               T* __restrict__ v, T* __restrict__ q, int bulk) {
  extern __shared__ __align__(128) unsigned char csr_sm[];
  T* sw = reinterpret_cast<T*>(csr_sm);  // [PC] each, PC a multiple of 4
  T* sv = sw + PC;
  T* sq = sv + PC;
  int32_t* sc = reinterpret_cast<int32_t*>(q ? sq + PC : sq);
  int r = blockIdx.x, first = 0;
  if (r >= rows) {
    const int x = r - rows;
    if (x >= *nextra) return;
    r = extra[x].row;
    first = extra[x].place * chunk;
  }
  const int c0 = blockIdx.y * PC, nc = min(PC, P - c0);
  const int words = ((q ? 3 : 2) * (int)sizeof(T) + 4) * PC / 16;
  for (int e = threadIdx.x; e < words; e += CSR_NT)
    reinterpret_cast<int4*>(csr_sm)[e] = make_int4(0, 0, 0, 0);
  constexpr int NW = CSR_NT / 32;
  const int all = rowcount[r], last = first + min(chunk, all - first);
  const int lane = threadIdx.x & 31, take = min(32, (last - first + NW - 1) / NW);
  const int32_t* lst = list + start[r];
  __syncthreads();
  for (int b = first + (int)(threadIdx.x >> 5) * take; b < last; b += NW * take) {
    int j = -1, lo = 0, ni = 0;
    double rj = 0.0, wj = 0.0;
    if (lane < take && b + lane < last) {
      j = lst[b + lane];
      const ObsRec o = rec[j];
      rj = o.r, lo = o.lo, ni = o.ni;
      wj = wt[j];
    }
    int end = ni;  // of the lane's pairs among the warp's
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += x;
    }
    const int total = __shfl_sync(0xffffffffu, end, 31);
    for (int p0 = 0; p0 < total; p0 += 32) {
      const int p = p0 + lane;
      int i = 0;  // pair p's observation: as many as end at or before p
#pragma unroll
      for (int step = 16; step > 0; step >>= 1)
        if (__shfl_sync(0xffffffffu, end, i + step - 1) <= p) i += step;
      const int l = __shfl_sync(0xffffffffu, lo + ni - end, i) + p;
      const int self = __shfl_sync(0xffffffffu, j, i);
      const double ri = __shfl_sync(0xffffffffu, rj, i), wi = __shfl_sync(0xffffffffu, wj, i);
      if (p >= total || l == self) continue;
      const int c = ob[l] - c0;
      if (c < 0 || c >= nc) continue;
      const double prod = ri * rec[l].r;
      atomicAdd(sc + c, 1);
      atomicAdd(sw + c, (T)wi);
      atomicAdd(sv + c, (T)(wi * prod));
      if (q) atomicAdd(sq + c, (T)(wi * prod * prod));
    }
  }
  const size_t o = (size_t)r * P + c0;
  if (all > chunk) {
    __syncthreads();
    for (int c = threadIdx.x; c < nc; c += CSR_NT) {
      if (sc[c] == 0) continue;
      atomicAdd(cnt + o + c, sc[c]);
      atomicAdd(w + o + c, sw[c]);
      atomicAdd(v + o + c, sv[c]);
      if (q) atomicAdd(q + o + c, sq[c]);
    }
    return;
  }
  if (bulk) {  // every thread's sums visible to the copies, which one thread issues
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
      auto put = [&](void* dst, const void* src, size_t bytes) {
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
                     "r"((uint32_t)__cvta_generic_to_shared(src)), "r"((uint32_t)bytes)
                     : "memory");
      };
      put(cnt + o, sc, sizeof(int32_t) * nc);
      put(w + o, sw, sizeof(T) * nc);
      put(v + o, sv, sizeof(T) * nc);
      if (q) put(q + o, sq, sizeof(T) * nc);
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }
    return;
  }
  __syncthreads();
  for (int c = threadIdx.x; c < nc; c += CSR_NT) {
    cnt[o + c] = sc[c];
    w[o + c] = sw[c];
    v[o + c] = sv[c];
    if (q) q[o + c] = sq[c];
  }
}


// ---------------------------------------------------------------------------
// FP32 covariance bins of gridded data, split by folds, on the tensor cores.
// Subjects with N_i >= 2 are put in fold order (stable).  With w_i = 1/(N_i(N_i - 1)), M the
// masks and R the responses (zero where unobserved), each fold's
//   C = M'M,  W = M'(w M),  V = X'X with X = sqrt(w) R,  Q = Z'Z with Z = sqrt(w) R^2
// are computed 128 x 128 outputs per block, for the tile pairs on and above the diagonal; the
// tile below is written as the transpose (all four are symmetric).
//
// FP32 from BF16 products: an FP32 number is exactly the sum of three BF16 ones (hi, mid, lo:
// 8 bits each), a product of BF16 numbers is exact, and X'X keeps the six of the nine part
// products that are above 2^-25 of the whole (mid lo, lo mid and lo lo are below it); w M is
// three products with the exact 0/1 plane, M'M one.  The tensor cores' accumulator cuts
// addends off instead of rounding them, a bias that would grow with the sum, so each run of 16
// subjects is accumulated from zero, smallest parts first, and added to the FP32 sums by
// ordinary additions: 4 additions beside 24 tensor instructions.  Against 64 bits the bins are
// closer than those of FP32 multiply-adds, whose chains are 16 times as long.
//
// These are warp-level products (mma.sync, 0.60 PFLOP/s measured here): tcgen05 is three times
// as fast, but its sums stay in tensor memory over many steps.  64 x 64, n = 1000, 5 folds
// (0.27 TFLOP of part products, 1.34 GB written): 808 us, half of it at the tensor rate, the rest
// the outputs and the stages' first loads (200 subjects a fold); the FP32 multiply-adds that this
// replaces took 1480 us at 58 % of their peak.
// ---------------------------------------------------------------------------
constexpr int FG_T = 128;            // output tile edge
constexpr int FG_K = 32;             // subjects per pipeline stage
constexpr int FG_NT = 256;           // threads: 8 warps of 64 x 32 outputs
constexpr int FG_LD = FG_T + 8;      // row pitch of a staged tile: ldmatrix without conflicts
constexpr int FG_PLANES = 7;         // M, X (3 parts), Z (3 parts)
constexpr int FG_TILE = FG_K * FG_LD;  // BF16 numbers of a staged tile
constexpr size_t FG_SMEM = 2ull * 6 * FG_TILE * 2;  // 2 stages of 2 x 3 tiles
constexpr int FG_OLD = FG_T + 1;     // row pitch of the output tile
static_assert(FG_SMEM >= sizeof(float) * FG_T * FG_OLD, "output tile in the stages");

__device__ __forceinline__ int fold_slot(int i, int F, const int32_t* __restrict__ fold,
                                         const int32_t* __restrict__ Ni, int* err) {
  if (Ni[i] < 2) return -1;  // no pairs
  if (!fold) return 0;
  const int f = fold[i];
  if (f < 0 || f >= F) {
    atomicExch(err, DERR_BOUNDS);
    return -1;
  }
  return f;
}

// Stable fold order (one block of 1024 threads): order[fstart[f] + r] is the r-th
// subject of fold f in index order; fstart[F] is the number of subjects kept.
__global__ void __launch_bounds__(1024)
    k_fold_order(int n, int F, const int32_t* __restrict__ fold, const int32_t* __restrict__ Ni,
                 int32_t* __restrict__ order, int32_t* __restrict__ fstart, int* err) {
  __shared__ int fcount[64];
  __shared__ int wpre[32][64];  // per warp and fold: count, then running position
  __shared__ int base[64];
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  if (tid < 64) fcount[tid] = 0;
  __syncthreads();
  for (int i = tid; i < n; i += 1024) {
    const int f = fold_slot(i, F, fold, Ni, err);
    if (f >= 0) atomicAdd(&fcount[f], 1);
  }
  __syncthreads();
  if (tid == 0) {
    int s = 0;
    for (int f = 0; f < F; ++f) {
      base[f] = s;
      fstart[f] = s;
      s += fcount[f];
    }
    fstart[F] = s;
  }
  __syncthreads();
  for (int c0 = 0; c0 < n; c0 += 1024) {
    for (int e = tid; e < 32 * 64; e += 1024) (&wpre[0][0])[e] = 0;
    __syncthreads();
    const int i = c0 + tid;
    const int f = i < n ? fold_slot(i, F, fold, Ni, err) : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, f);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    if (f >= 0 && rank == 0) wpre[wp][f] = __popc(peers);
    __syncthreads();
    if (tid < F) {  // exclusive prefix over the warps, fold by fold
      int run = base[tid];
      for (int w2 = 0; w2 < 32; ++w2) {
        const int c = wpre[w2][tid];
        wpre[w2][tid] = run;
        run += c;
      }
      base[tid] = run;
    }
    __syncthreads();
    if (f >= 0) order[wpre[wp][f] + rank] = i;
    __syncthreads();
  }
}

// x = p[0] + p[1] + p[2] exactly (finite x above 2^-110); what is not finite stays in p[0]
__device__ __forceinline__ void split3(float x, __nv_bfloat16* p) {
  p[0] = __float2bfloat16_rn(x);
  p[1] = p[2] = __float2bfloat16_rn(0.f);
  if (!isfinite(x)) return;
  if (!isfinite(__bfloat162float(p[0])))  // rounded past the largest: cut off instead
    p[0] = __ushort_as_bfloat16((unsigned short)(__float_as_uint(x) >> 16));
  const float r1 = x - __bfloat162float(p[0]);
  p[1] = __float2bfloat16_rn(r1);
  p[2] = __float2bfloat16_rn(r1 - __bfloat162float(p[1]));
}

// Operand rows in fold order, FO_ROWS rows by 512 columns a block, 4 columns a thread; rows
// past fstart[F] are left alone (the Gram kernel never reads them).  The residuals are
// float-float (FP64 subtractions and conversions of every entry took most of the 45 us that
// this pass had at n = 1000, P = 4096), mu split once per FO_ROWS subjects.
constexpr int FO_ROWS = 8;
__global__ void __launch_bounds__(128)
    k_fold_operands(int n, int P, int Ps, int F, const void* __restrict__ y, int y_prec,
                    const uint8_t* __restrict__ mask, const int32_t* __restrict__ Ni,
                    const double* __restrict__ mu, int mode, const int32_t* __restrict__ order,
                    const int32_t* __restrict__ fstart, __nv_bfloat16* __restrict__ X,
                    float* __restrict__ ws) {
  __shared__ int who[FO_ROWS];
  __shared__ ff::F2 root[FO_ROWS];
  const int k0 = blockIdx.x * FO_ROWS, kn = min(FO_ROWS, fstart[F] - k0);
  if (kn <= 0) return;
  if ((int)threadIdx.x < kn) {
    const int i = order[k0 + threadIdx.x];
    const double N = (double)Ni[i], w = 1.0 / (N * (N - 1.0)), s = sqrt(w);
    who[threadIdx.x] = i;
    root[threadIdx.x] = {(float)s, (float)(s - (double)(float)s)};
    if (blockIdx.y == 0) ws[k0 + threadIdx.x] = (float)w;
  }
  __syncthreads();
  const int p0 = (blockIdx.y * 128 + threadIdx.x) * 4;
  if (p0 >= Ps) return;
  double md[4] = {0.0, 0.0, 0.0, 0.0};
  ff::F2 m2[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (mode == FPCA_COV_RESIDUAL && p0 + u < P) md[u] = mu[p0 + u];
    m2[u] = {(float)md[u], (float)(md[u] - (double)(float)md[u])};
  }
  const size_t plane = (size_t)n * Ps;
  for (int r = 0; r < kn; ++r) {
    __align__(8) __nv_bfloat16 o[FG_PLANES][4];
    const ff::F2 s = root[r];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t at = (size_t)who[r] * P + p0 + u;
      float one = 0.f, x = 0.f, z = 0.f;
      if (p0 + u < P && (!mask || mask[at])) {
        ff::F2 d;
        if (y_prec == FPCA_F64) {
          const double dd = static_cast<const double*>(y)[at] - md[u];
          d = {(float)dd, 0.f};
          if (isfinite(d.hi)) d.lo = (float)(dd - (double)d.hi);
        } else {
          const float v = static_cast<const float*>(y)[at];
          const ff::F2 t = ff::two_sum(v, -m2[u].hi);
          d = isfinite(t.hi) ? ff::fast_two_sum(t.hi, t.lo - m2[u].lo) : ff::make(t.hi);
        }
        one = 1.f;
        x = ff::mul(s, d).hi;
        z = ff::mul(s, ff::mul(d, d)).hi;
        if (!isfinite(x)) x = s.hi * d.hi;  // the corrections of an overflow are not numbers
        if (!isfinite(z)) z = s.hi * (d.hi * d.hi);
      }
      __nv_bfloat16 px[3], pz[3];
      split3(x, px);
      split3(z, pz);
      o[0][u] = __float2bfloat16_rn(one);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        o[1 + c][u] = px[c];
        o[4 + c][u] = pz[c];
      }
    }
#pragma unroll
    for (int c = 0; c < FG_PLANES; ++c)
      *reinterpret_cast<uint2*>(X + c * plane + (size_t)(k0 + r) * Ps + p0) =
          *reinterpret_cast<const uint2*>(o[c]);
  }
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
               "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// the same from zero
__device__ __forceinline__ void mma_bf16_zero(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                              uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%10,%10,%10,%10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// Output tile of one fold and plane over stages of FG_K subjects.  KIND 0: M'M (exact, so
// accumulated in place); 1: M'(w M); 2: the six part products of X'X.  A warp's 64 x 32
// outputs are 4 x 4 tensor tiles; KIND 2 takes 16 columns at a time, since all 32 would not
// leave the registers for two blocks an SM.  32 x 32 a warp, with 32 columns at a time but a
// 64 x 128 tile a block, reads half as much again from L2, which carries 6.9 TB/s then, and was
// slower (1.00 ms against 0.96), also with the next plane's first stage behind the outputs' stores.
template <int KIND>
__device__ __forceinline__ void fold_tile(__nv_bfloat16* st, __nv_bfloat16 (*sw)[3][FG_K],
                                          const __nv_bfloat16* __restrict__ src, size_t plane,
                                          int Ps, const float* __restrict__ ws, int p0, int q0,
                                          int k0, int k1, float (&acc)[4][4][4]) {
  constexpr int NP = KIND == 2 ? 3 : 1;
  constexpr int NH = KIND == 2 ? 1 : 2;  // 16-column halves at a time
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = (warp & 1) * 64, wn = (warp >> 1) * 32;
  const int lr = tid >> 4, lc = (tid & 15) * 8;  // this thread's 16 bytes of a tile: rows lr, lr + 16
  const uint32_t sdst = smem_addr(st + lr * FG_LD + lc);
  auto load = [&](int s, int kb) {
    const bool ok0 = kb + lr < k1, ok1 = kb + lr + 16 < k1;
    const size_t o0 = (size_t)(ok0 ? kb + lr : k0) * Ps + lc;
    const size_t o1 = (size_t)(ok1 ? kb + lr + 16 : k0) * Ps + lc;
#pragma unroll
    for (int c = 0; c < 2 * NP; ++c) {  // the parts of rows p0.., then of columns q0..
      const __nv_bfloat16* pl = src + (c % NP) * plane + (c < NP ? p0 : q0);
      const uint32_t d = sdst + 2 * (s * 6 + c) * FG_TILE;
      cp_async16(d, pl + o0, ok0);
      cp_async16(d + 2 * 16 * FG_LD, pl + o1, ok1);
    }
    if (KIND == 1 && tid < FG_K) {
      __nv_bfloat16 w[3];
      split3(kb + tid < k1 ? ws[kb + tid] : 0.f, w);
      for (int c = 0; c < 3; ++c) sw[s][c][tid] = w[c];
    }
  };
  const int nchunk = (k1 - k0 + FG_K - 1) / FG_K;
  if (nchunk > 0) load(0, k0);
  cp_async_commit();
  for (int ch = 0; ch < nchunk; ++ch) {
    const int s = ch & 1;
    if (ch + 1 < nchunk) load(s ^ 1, k0 + (ch + 1) * FG_K);
    cp_async_commit();
    cp_async_wait1();
    __syncthreads();
    const uint32_t base = smem_addr(st + s * 6 * FG_TILE);
    // this lane's row of the four 8 x 8 matrices that ldmatrix reads, for both operands
    const uint32_t la = base + 2 * (((lane >> 4) * 8 + (lane & 7)) * FG_LD + wm + ((lane >> 3) & 1) * 8);
    const uint32_t lb = base + 2 * (NP * FG_TILE + (((lane >> 3) & 1) * 8 + (lane & 7)) * FG_LD + wn +
                                    (lane >> 4) * 8);
    // the second 16 subjects of the last stage may be beyond the fold
    const int ksn = k0 + ch * FG_K + 16 < k1 ? 2 : 1;
#pragma unroll 1
    for (int ks = 0; ks < ksn; ++ks) {
      __nv_bfloat162 wk[3][2];
      if constexpr (KIND == 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int e = 0; e < 2; ++e)
            wk[c][e] = *reinterpret_cast<const __nv_bfloat162*>(&sw[s][c][ks * 16 + 8 * e + 2 * (lane & 3)]);
      }
#pragma unroll
      for (int h0 = 0; h0 < 2; h0 += NH) {
        uint32_t b[NP][NH][4];
#pragma unroll
        for (int c = 0; c < NP; ++c)
#pragma unroll
          for (int h = 0; h < NH; ++h)
            ldsm4t(b[c][h], lb + 2 * (c * FG_TILE + ks * 16 * FG_LD + (h0 + h) * 16));
#pragma unroll
        for (int mi = 0; mi < 4; ++mi) {
          uint32_t a[NP][4];
#pragma unroll
          for (int c = 0; c < NP; ++c)
            ldsm4t(a[c], la + 2 * (c * FG_TILE + ks * 16 * FG_LD + mi * 16));
          float t[2 * NH][4];
          auto first = [&](const uint32_t (&x)[4], int cb) {
#pragma unroll
            for (int ni = 0; ni < 2 * NH; ++ni)
              mma_bf16_zero(t[ni], x, b[cb][ni >> 1][2 * (ni & 1)], b[cb][ni >> 1][2 * (ni & 1) + 1]);
          };
          auto part = [&](const uint32_t (&x)[4], int cb) {
#pragma unroll
            for (int ni = 0; ni < 2 * NH; ++ni)
              mma_bf16(t[ni], x, b[cb][ni >> 1][2 * (ni & 1)], b[cb][ni >> 1][2 * (ni & 1) + 1]);
          };
          if constexpr (KIND == 0) {
#pragma unroll
            for (int ni = 0; ni < 4; ++ni)
              mma_bf16(acc[mi][ni], a[0], b[0][ni >> 1][2 * (ni & 1)], b[0][ni >> 1][2 * (ni & 1) + 1]);
          } else {
            if constexpr (KIND == 2) {
              first(a[2], 0);
              part(a[0], 2);
              part(a[1], 1);
              part(a[1], 0);
              part(a[0], 1);
              part(a[0], 0);
            } else {
#pragma unroll
              for (int c = 2; c >= 0; --c) {
                uint32_t x[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const __nv_bfloat162 v =
                      __hmul2(*reinterpret_cast<const __nv_bfloat162*>(&a[0][e]), wk[c][e >> 1]);
                  x[e] = *reinterpret_cast<const uint32_t*>(&v);
                }
                if (c == 2)
                  first(x, 0);
                else
                  part(x, 0);
              }
            }
#pragma unroll
            for (int ni = 0; ni < 2 * NH; ++ni)
#pragma unroll
              for (int e = 0; e < 4; ++e) acc[mi][2 * h0 + ni][e] += t[ni][e];
          }
        }
      }
    }
    __syncthreads();  // the stage is overwritten by the load after next
  }
}

// One entry of X'X from the whole numbers, where a part product was no number (overflows,
// infinities and NaN among the observations).
__device__ __noinline__ float fold_entry(const __nv_bfloat16* __restrict__ src, size_t plane, int Ps,
                                         int p, int q, int k0, int k1) {
  float x = 0.f;
  for (int k = k0; k < k1; ++k) {
    const __nv_bfloat16 *a = src + (size_t)k * Ps + p, *b = src + (size_t)k * Ps + q;
    const float av = __bfloat162float(a[0]) + (__bfloat162float(a[plane]) + __bfloat162float(a[2 * plane]));
    const float bv = __bfloat162float(b[0]) + (__bfloat162float(b[plane]) + __bfloat162float(b[2 * plane]));
    x = fmaf(av, bv, x);
  }
  return x;
}

// blockIdx.x: tile pair (bi <= bj), y: fold, z: Q, V, W, C, the costly ones first.  vec2: P even
// and the outputs aligned to 8 bytes.
__global__ void __launch_bounds__(FG_NT, 2)
    k_fold_gram(int n, int P, int Ps, const __nv_bfloat16* __restrict__ X,
                const float* __restrict__ ws, const int32_t* __restrict__ fstart,
                const int2* __restrict__ pairs, int32_t* __restrict__ cnt, float* __restrict__ w,
                float* __restrict__ v, float* __restrict__ q, int with_q, int vec2) {
  extern __shared__ __align__(16) __nv_bfloat16 fst[];
  __shared__ __align__(4) __nv_bfloat16 sw[2][3][FG_K];
  const int2 pr = pairs[blockIdx.x];
  const int f = blockIdx.y, z = with_q ? (blockIdx.z + 3) & 3 : blockIdx.z;  // 3 Q, 0 V, 1 W, 2 C
  const int k0 = fstart[f], k1 = fstart[f + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int p0 = pr.x * FG_T, q0 = pr.y * FG_T;
  const size_t plane = (size_t)n * Ps;
  const __nv_bfloat16* src = X + (z == 0 ? 1 : z == 3 ? 4 : 0) * plane;
  float acc[4][4][4] = {};
  if (z == 0 || z == 3)
    fold_tile<2>(fst, sw, src, plane, Ps, ws, p0, q0, k0, k1, acc);
  else if (z == 1)
    fold_tile<1>(fst, sw, src, plane, Ps, ws, p0, q0, k0, k1, acc);
  else
    fold_tile<0>(fst, sw, src, plane, Ps, ws, p0, q0, k0, k1, acc);
  const size_t fo = (size_t)f * P * P;
  uint32_t* out = reinterpret_cast<uint32_t*>(z == 0 ? v : z == 1 ? w : z == 3 ? q : (float*)cnt) + fo;
  auto bits = [&](float x) { return z == 2 ? (uint32_t)__float2int_rn(x) : __float_as_uint(x); };
  // the tile from the registers, whole sectors of its rows; its transpose by whole lines through
  // shared memory.  Streaming stores: not read here again, so that the operands stay in L2.
  const bool diag = p0 == q0, inside = p0 + FG_T <= P && q0 + FG_T <= P;
  float* T = reinterpret_cast<float*>(fst);
  bool odd = false;
#pragma unroll
  for (int mi = 0; mi < 4; ++mi)
#pragma unroll
    for (int ni = 0; ni < 4; ++ni)
#pragma unroll
      for (int e = 0; e < 4; e += 2) {
        const int r = (warp & 1) * 64 + mi * 16 + (lane >> 2) + 4 * e;
        const int c = (warp >> 1) * 32 + ni * 8 + 2 * (lane & 3);
        float x0 = acc[mi][ni][e], x1 = acc[mi][ni][e + 1];
        if (diag && r == c) x0 = 0.f;  // only pairs of an observation with itself
        if (diag && r == c + 1) x1 = 0.f;
        odd |= !isfinite(x0) || !isfinite(x1);
        T[r * FG_OLD + c] = x0;
        T[r * FG_OLD + c + 1] = x1;
        uint32_t* o = out + (size_t)(p0 + r) * P + q0 + c;
        if (inside && vec2) {
          __stcs(reinterpret_cast<uint2*>(o), make_uint2(bits(x0), bits(x1)));
        } else if (p0 + r < P) {
          if (q0 + c < P) __stcs(o, bits(x0));
          if (q0 + c + 1 < P) __stcs(o + 1, bits(x1));
        }
      }
  odd = __syncthreads_or(odd);
  if (!diag)
    for (int c = warp; c < FG_T && q0 + c < P; c += FG_NT / 32) {
      uint32_t* o = out + (size_t)(q0 + c) * P + p0 + lane;
#pragma unroll
      for (int j = 0; j < FG_T / 32; ++j)
        if (p0 + lane + 32 * j < P) __stcs(o + 32 * j, bits(T[(lane + 32 * j) * FG_OLD + c]));
    }
  if (odd && (z == 0 || z == 3)) {  // overflows, infinities, NaN
    __syncthreads();                // the transposed entries are written again here
    for (int e = tid; e < FG_T * FG_T; e += FG_NT) {
      const int r = p0 + e / FG_T, c = q0 + e % FG_T;
      if (r >= P || c >= P || isfinite(T[e / FG_T * FG_OLD + e % FG_T])) continue;
      const uint32_t x = __float_as_uint(fold_entry(src, plane, Ps, r, c, k0, k1));
      out[(size_t)r * P + c] = x;
      if (!diag) out[(size_t)c * P + r] = x;
    }
  }
}

}  // namespace

fpca_status launch_subject_counts_dense(fpca_ctx* ctx, int n, int P, const uint8_t* mask,
                                        int32_t* Ni) {
  k_subject_counts<<<(n + 7) / 8, 256, 0, ctx->stream>>>(n, P, mask, Ni);
  FPCA_LAUNCHED(ctx, "subject_counts");
  return FPCA_OK;
}

fpca_status launch_bin_mean_dense(fpca_ctx* ctx, int n, int P, const void* y, int y_prec,
                                  const uint8_t* mask, const int32_t* Ni, int32_t* cnt,
                                  double* w, double* v, double* v2) {
  if (y_prec == FPCA_F64)
    k_bin_mean_dense<double><<<(P + 31) / 32, dim3(32, MB_SLICES), 0, ctx->stream>>>(
        n, P, static_cast<const double*>(y), mask, Ni, cnt, w, v, v2);
  else
    k_bin_mean_dense<float><<<(P + 31) / 32, dim3(32, MB_SLICES), 0, ctx->stream>>>(
        n, P, static_cast<const float*>(y), mask, Ni, cnt, w, v, v2);
  FPCA_LAUNCHED(ctx, "bin_mean_dense");
  return FPCA_OK;
}

fpca_status launch_bin_mean_sparse(fpca_ctx* ctx, int n, const fpca_grid* g, const int64_t* offs,
                                   const double* t, const double* y, int32_t* cnt, double* w,
                                   double* v, double* v2) {
  const int P = grid_P(g);
  int64_t Nobs = 0;
  if (fpca_no_capture(ctx, "reading offs[n] of scattered data") != FPCA_OK) return FPCA_E_UNSUPPORTED;
  cudaError_t e = cudaMemcpyAsync(&Nobs, offs + n, sizeof(int64_t), cudaMemcpyDeviceToHost,
                                  ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) return fpca_fail(ctx, FPCA_E_CUDA, "reading offs[n]: %s", cudaGetErrorString(e));
  if (Nobs < 0) return fpca_fail(ctx, FPCA_E_INVALID_ARG, "offs[n] = %lld", (long long)Nobs);
  cudaMemsetAsync(cnt, 0, sizeof(int32_t) * P, ctx->stream);
  cudaMemsetAsync(w, 0, sizeof(double) * P, ctx->stream);
  cudaMemsetAsync(v, 0, sizeof(double) * P, ctx->stream);
  if (v2) cudaMemsetAsync(v2, 0, sizeof(double) * P, ctx->stream);
  k_bin_mean_sparse<<<(n + 127) / 128, 128, 0, ctx->stream>>>(
      n, (long long)Nobs, g->d, g->m[0], g->d > 1 ? g->m[1] : 1, g->d > 2 ? g->m[2] : 1, offs, t,
      y, cnt, w, v, v2, ctx->d_err);
  FPCA_LAUNCHED(ctx, "bin_mean_sparse");
  return FPCA_OK;
}

fpca_status launch_cov_operands_bf16(fpca_ctx* ctx, int n, int P, int Kpad, const void* y,
                                     int y_prec, const uint8_t* mask, const int32_t* Ni,
                                     const double* mu, int mode, uint16_t* ops) {
  if (Kpad % 64 != 0) return fpca_fail(ctx, FPCA_E_INVALID_ARG, "Kpad = %d", Kpad);
  dim3 grid((P + 31) / 32, Kpad / 64);
  __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(ops);
  if (y_prec == FPCA_F64)
    k_cov_operands_bf16<double><<<grid, dim3(32, 8), 0, ctx->stream>>>(
        n, P, Kpad, static_cast<const double*>(y), mask, Ni, mu, mode, o2);
  else
    k_cov_operands_bf16<float><<<grid, dim3(32, 8), 0, ctx->stream>>>(
        n, P, Kpad, static_cast<const float*>(y), mask, Ni, mu, mode, o2);
  FPCA_LAUNCHED(ctx, "cov_operands_bf16");
  return FPCA_OK;
}

fpca_status launch_cov_dense_f64(fpca_ctx* ctx, int n, int P, const void* y, int y_prec,
                                 const uint8_t* mask, const int32_t* Ni, const double* mu,
                                 int mode, int32_t* cnt, double* w, double* v) {
  const int nt = (P + CD_T - 1) / CD_T;
  k_cov_dense_f64<<<(unsigned)((long long)nt * (nt + 1) / 2), CD_T * CD_T, 0, ctx->stream>>>(
      n, P, nt, y, y_prec, mask, Ni, mu, mode, cnt, w, v);
  FPCA_LAUNCHED(ctx, "cov_dense_f64");
  return FPCA_OK;
}

fpca_status launch_cov_sparse(fpca_ctx* ctx, int n, const fpca_grid* g, const int64_t* offs,
                              const double* t, const double* y, const double* mu, int mode,
                              const int32_t* fold, int nfold, int prec, int32_t* cnt, void* w,
                              void* v, void* q) {
  const int P = grid_P(g);
  const int F = nfold > 0 ? nfold : 1;
  // total observation count (offs[n]) is needed on the host to size the launch
  int64_t Nobs = 0;
  if (fpca_no_capture(ctx, "reading offs[n] of scattered data") != FPCA_OK) return FPCA_E_UNSUPPORTED;
  cudaError_t e = cudaMemcpyAsync(&Nobs, offs + n, sizeof(int64_t), cudaMemcpyDeviceToHost,
                                  ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) return fpca_fail(ctx, FPCA_E_CUDA, "reading offs[n]: %s", cudaGetErrorString(e));
  if (Nobs < 0 || Nobs > (1ll << 31))
    return fpca_fail(ctx, FPCA_E_INVALID_ARG, "offs[n] = %lld out of range", (long long)Nobs);
  if ((long long)P * F > 0x7fffffffll)
    return fpca_fail(ctx, FPCA_E_UNSUPPORTED, "%d bins x %d folds", P, F);
  const int rows = P * F;
  const size_t N = (size_t)Nobs;
  // columns per CTA: at most 64 KB (FP32) or 56 KB (FP64) of sums, so that three CTAs share
  // an SM and one's copies out overlap the others' sums
  const int PC = std::min(prec == FPCA_F64 ? 2048 : 4096, (P + 3) / 4 * 4);
  const int ncol = (P + PC - 1) / PC;
  // chunks: no row is longer than what gives every SM a dozen (fewer, and the last to start hold
  // up the call; many more, and rows that would not need it are cleared and added)
  const int chunk = (int)std::max<long long>(CSR_CHUNK, Nobs * ncol / (12ll * ctx->num_sms));
  const int nx = (int)(Nobs / chunk);  // further chunks at most
  // a launch of its own for the counts pays where a counter would take many atomics
  const bool count = rows <= RC_ROWS && Nobs > 64ll * rows;
  void* ws = fpca_workspace(ctx, WsCarve::round(4 * N) * 4 + WsCarve::round(sizeof(ObsRec) * N) +
                                     WsCarve::round(sizeof(double) * N) +
                                     WsCarve::round(sizeof(RowChunk) * (size_t)nx) +
                                     WsCarve::round(4 * (size_t)rows) * 2 + 4096);
  if (!ws) return fpca_fail(ctx, FPCA_E_OOM, "workspace");
  WsCarve carve(ws);
  int32_t* ob = carve.take<int32_t>(N);
  // row, and the rows' counts behind it: cleared together ([rows]: the list's length)
  int32_t* row = carve.take<int32_t>(N + (size_t)rows + 2);
  int32_t* rowcount = row + N;
  int32_t* rank = carve.take<int32_t>(N);
  int32_t* list = carve.take<int32_t>(N);
  ObsRec* rec = carve.take<ObsRec>(N);
  double* wt = carve.take<double>(N);
  RowChunk* extra = carve.take<RowChunk>(nx);
  int32_t* nextra = rowcount + rows + 1;
  int32_t* start = carve.take<int32_t>(rows);
  cudaMemsetAsync(row, 0, sizeof(int32_t) * (N + (size_t)rows + 2), ctx->stream);
  if (Nobs > 0) {
    k_obs_rows<<<(int)(((long long)n * OBS_LANES + 255) / 256), 256, 0, ctx->stream>>>(
        n, Nobs, g->d, g->m[0], g->d > 1 ? g->m[1] : 1, g->d > 2 ? g->m[2] : 1, P, offs, t, y, mu,
        mode, fold, nfold, ob, rec, wt, row, rowcount, count ? nullptr : rank, ctx->d_err);
    FPCA_LAUNCHED(ctx, "obs_rows");
    if (count) {
      const long long per = RC_NT * RC_PER;
      k_row_count<<<(int)((Nobs + per - 1) / per), RC_NT, 0, ctx->stream>>>(Nobs, rows, row,
                                                                            rowcount, rank);
      FPCA_LAUNCHED(ctx, "row_count");
    }
  }
  k_row_starts<<<(rows + 255) / 256, 256, 0, ctx->stream>>>(rows, chunk, rowcount, start,
                                                            rowcount + rows, nextra, extra);
  FPCA_LAUNCHED(ctx, "row_starts");
  if (Nobs > 0) {
    const int fill = (int)((Nobs + 255) / 256);
    k_row_fill<<<fill + nx, 256, 0, ctx->stream>>>(Nobs, fill, row, start, rank, list, P,
                                                   prec == FPCA_F64 ? 8 : 4, nextra, extra, cnt, w,
                                                   v, q);
    FPCA_LAUNCHED(ctx, "row_fill");
  }
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const int bulk = (P % 4 == 0 && al16(cnt) && al16(w) && al16(v) && (!q || al16(q))) ? 1 : 0;
  auto launch = [&](auto kern, auto* pw, auto* pv, auto* pq) -> fpca_status {
    const size_t sm = (size_t)PC * ((pq ? 3 : 2) * sizeof(*pw) + 4);
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    kern<<<dim3(rows + nx, ncol), CSR_NT, sm, ctx->stream>>>(rows, P, PC, chunk, rowcount, start,
                                                             list, ob, rec, wt, nextra, extra, cnt,
                                                             pw, pv, pq, bulk);
    FPCA_LAUNCHED(ctx, "cov_rows");
    return FPCA_OK;
  };
  if (prec == FPCA_F64)
    return launch(k_cov_rows<double>, static_cast<double*>(w), static_cast<double*>(v),
                  static_cast<double*>(q));
  return launch(k_cov_rows<float>, static_cast<float*>(w), static_cast<float*>(v),
                static_cast<float*>(q));
}

fpca_status launch_cov_dense_folds(fpca_ctx* ctx, int n, int P, const void* y, int y_prec,
                                   const uint8_t* mask, const double* mu, int mode,
                                   const int32_t* fold, int nfold, int32_t* cnt, float* w,
                                   float* v, float* q) {
  const int F = nfold > 0 ? nfold : 1;
  if (n == 0) {  // no subjects: every bin is empty
    const size_t PPF = (size_t)P * P * F;
    cudaMemsetAsync(cnt, 0, sizeof(int32_t) * PPF, ctx->stream);
    cudaMemsetAsync(w, 0, sizeof(float) * PPF, ctx->stream);
    cudaMemsetAsync(v, 0, sizeof(float) * PPF, ctx->stream);
    if (q) cudaMemsetAsync(q, 0, sizeof(float) * PPF, ctx->stream);
    return fpca_check_launch(ctx, "cov_fold_gram memset");
  }
  const int Ps = (P + FG_T - 1) / FG_T * FG_T;
  const int nt = Ps / FG_T;
  const size_t need = WsCarve::round(sizeof(int32_t) * (size_t)n) * 2 +
                      WsCarve::round(sizeof(int32_t) * 65) +
                      WsCarve::round(sizeof(__nv_bfloat16) * FG_PLANES * (size_t)n * Ps) +
                      WsCarve::round(sizeof(float) * (size_t)n) +
                      WsCarve::round(sizeof(int2) * (size_t)nt * (nt + 1) / 2) + 2048;
  void* wsp = fpca_workspace(ctx, need);
  if (!wsp) return fpca_fail(ctx, FPCA_E_OOM, "workspace (%zu bytes)", need);
  WsCarve carve(wsp);
  int32_t* Ni = carve.take<int32_t>(n);
  int32_t* order = carve.take<int32_t>(n);
  int32_t* fstart = carve.take<int32_t>(65);
  __nv_bfloat16* X = carve.take<__nv_bfloat16>(FG_PLANES * (size_t)n * Ps);
  float* wsub = carve.take<float>(n);
  int2* pairs = carve.take<int2>((size_t)nt * (nt + 1) / 2);
  std::vector<int2> ph;
  ph.reserve((size_t)nt * (nt + 1) / 2);
  for (int bi = 0; bi < nt; ++bi)
    for (int bj = bi; bj < nt; ++bj) ph.push_back(make_int2(bi, bj));
  // pageable source: staged before the call returns (so not capturable)
  if (fpca_no_capture(ctx, "the fold-split binning of gridded data") != FPCA_OK)
    return FPCA_E_UNSUPPORTED;
  if (cudaMemcpyAsync(pairs, ph.data(), sizeof(int2) * ph.size(), cudaMemcpyHostToDevice,
                      ctx->stream) != cudaSuccess)
    return fpca_check_launch(ctx, "fold gram tile pairs");
  fpca_status s = launch_subject_counts_dense(ctx, n, P, mask, Ni);
  if (s != FPCA_OK) return s;
  k_fold_order<<<1, 1024, 0, ctx->stream>>>(n, F, nfold > 0 ? fold : nullptr, Ni, order, fstart,
                                            ctx->d_err);
  FPCA_LAUNCHED(ctx, "fold_order");
  k_fold_operands<<<dim3((n + FO_ROWS - 1) / FO_ROWS, (Ps + 511) / 512), 128, 0, ctx->stream>>>(
      n, P, Ps, F, y, y_prec, mask, Ni, mu, mode, order, fstart, X, wsub);
  FPCA_LAUNCHED(ctx, "fold_operands");
  const dim3 grid((unsigned)ph.size(), F, q ? 4 : 3);
  auto al8 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 7) == 0; };
  const int vec2 = P % 2 == 0 && al8(cnt) && al8(w) && al8(v) && al8(q);
  cudaFuncSetAttribute(k_fold_gram, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FG_SMEM);
  k_fold_gram<<<grid, FG_NT, FG_SMEM, ctx->stream>>>(n, P, Ps, X, wsub, fstart, pairs, cnt, w, v, q,
                                                     q ? 1 : 0, vec2);
  FPCA_LAUNCHED(ctx, "cov_fold_gram");
  return FPCA_OK;
}
