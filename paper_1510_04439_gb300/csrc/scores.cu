// Principal component scores, reconstruction and its error (Section 2.1, Section 4).
//
// PACE, Eq. (2.7): A_i = Lambda Phi_i' (Phi_i Lambda Phi_i' + sigma^2 I)^{-1} Y_i^C.
// By the push-through identity Lambda Phi' (Phi Lambda Phi' + sigma^2 I)^{-1} =
// (sigma^2 Lambda^{-1} + Phi'Phi)^{-1} Phi', each subject needs only the L x L
// system (sigma^2 Lambda^{-1} + Phi_i'Phi_i) A_i = Phi_i' Y_i^C instead of an
// N_i x N_i one.  Scattered data: one warp accumulates both sums over the subject's
// observations.  Gridded data: the Phi_i'Phi_i of all subjects are one integer
// matrix product on the tensor cores (k_pace_gram).  The systems are solved in
// float-float with one FP64 refinement (pace_solve).  Functions known on the grid
// are read at the bin of each observation (Section 3.2 binning).
//
// Scores by integration (dense data): A_il = dV sum over observed nodes of
// (Y_i - mu) phi_l; reconstruction X_i = mu + sum_l A_il phi_l at the nodes; the
// MISE of a reconstruction (Section 4) is the mean over subjects of the Riemann
// sum of (Xhat_i - X_i)^2.
//
// Arithmetic: the long sums run in FP32 with error-free transformations (the
// compensated dot product of Ogita, Rump and Oishi, "Accurate sum and dot
// product", 2005, on float-float inputs from ff.cuh): about FP64 accuracy at
// FP32 cost, since FP64 throughput on this GPU is 1/64 of FP32.  mu and phi are
// split into float-float once per call.
#include <algorithm>
#include <cmath>

#include <cuda_fp16.h>

#include "fpca_internal.cuh"
#include "ff.cuh"

namespace {

constexpr int SC_LMAX = 16;

struct ScGrid {
  int d, m[3], P;
};

__device__ __forceinline__ int sc_bin(const ScGrid& g, const double* t) {
  int b = 0;
  for (int k = 0; k < g.d; ++k) {
    const double x = floor(__dmul_rn(t[k], (double)g.m[k]));
    b = b * g.m[k] + (int)fmin(fmax(x, 0.0), (double)(g.m[k] - 1));
  }
  return b;
}

// Compensated accumulator: s + c is the running sum; each product a b of two
// float-float numbers enters through a two-product and a two-sum, and all the
// rounding errors are collected in c.
struct Acc {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add_prod(ff::F2 a, ff::F2 b) {
    const ff::F2 p = ff::two_prod(a.hi, b.hi);
    const ff::F2 t = ff::two_sum(s, p.hi);
    s = t.hi;
    c += t.lo + (p.lo + fmaf(a.hi, b.lo, a.lo * b.hi));
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

__device__ __forceinline__ ff::F2 split(double x) {
  const float hi = (float)x;
  return {hi, (float)(x - (double)hi)};
}

// y - m in float-float, y FP32 or FP64, m = mu as float-float
__device__ __forceinline__ ff::F2 centred(double y, ff::F2 m) {
  return split(y - ((double)m.hi + (double)m.lo));
}
__device__ __forceinline__ ff::F2 centred(float y, ff::F2 m) {
  const ff::F2 t = ff::two_sum(y, -m.hi);
  return ff::fast_two_sum(t.hi, t.lo - m.lo);
}
__device__ __forceinline__ ff::F2 centred(const void* y, int yprec, long long e, ff::F2 m) {
  return yprec == FPCA_F64 ? centred(static_cast<const double*>(y)[e], m)
                           : centred(static_cast<const float*>(y)[e], m);
}

// mu (row 0) and the first L eigenfunctions (rows 1..L) as float-float; bmax (L x gridDim.x, or
// NULL): each block's largest |phi_l|, rounded up, infinity if one is not finite.  For PACE (lam not
// NULL) prior[l] = sigma^2 / lambda_l, and prior[SC_LMAX] = 1 if sigma^2 >= 0 and every
// lambda > 0, else 0 (an FP64 division in every block of the later kernels took 3 us there).
__global__ void __launch_bounds__(256)
    k_split_ff(int P, const double* __restrict__ mu, const double* __restrict__ phi,
               float2* __restrict__ mu2, float2* __restrict__ phi2, float* __restrict__ bmax, int L,
               const double* __restrict__ lam, const double* __restrict__ sigma2p,
               double* __restrict__ prior) {
  __shared__ float wmax[8];
  if (lam && blockIdx.x == 0 && blockIdx.y == 0) {
    const double s2 = *sigma2p;
    const bool bad = !(s2 >= 0.0) || ((int)threadIdx.x < L && !(lam[threadIdx.x] > 0.0));
    if ((int)threadIdx.x < L) prior[threadIdx.x] = s2 / lam[threadIdx.x];
    const int any = __syncthreads_or(bad);
    if (threadIdx.x == 0) prior[SC_LMAX] = any ? 0.0 : 1.0;
  }
  const int l = (int)blockIdx.y - 1;
  const double* in = l < 0 ? mu : phi + (long long)l * P;
  float2* out = l < 0 ? mu2 : phi2 + (long long)l * P;
  float top = 0.f;
  for (long long e = blockIdx.x * 256 + threadIdx.x; e < P; e += gridDim.x * 256) {
    const ff::F2 v = split(in[e]);
    out[e] = make_float2(v.hi, v.lo);
    const float a = __double2float_ru(fabs(in[e]));
    top = isfinite(a) ? fmaxf(top, a) : INFINITY;
  }
  if (l < 0 || !bmax) return;
  for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = top;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) top = fmaxf(top, wmax[w]);
    bmax[(long long)l * gridDim.x + blockIdx.x] = top;
  }
}

// ---------------------------------------------------------------------------
// the L x L systems
// ---------------------------------------------------------------------------

// A a = b by Cholesky in FP64, in place; false if A is not positive definite.
__device__ bool solve_serial(double (*A)[SC_LMAX + 1], double* bb, int L) {
  for (int jj = 0; jj < L; ++jj) {
    double dj = A[jj][jj];
    for (int k = 0; k < jj; ++k) dj -= A[jj][k] * A[jj][k];
    if (!(dj > 0.0)) return false;
    const double ljj = sqrt(dj), il = 1.0 / ljj;
    A[jj][jj] = ljj;
    for (int r = jj + 1; r < L; ++r) {
      double v = A[r][jj];
      for (int k = 0; k < jj; ++k) v -= A[r][k] * A[jj][k];
      A[r][jj] = v * il;
    }
  }
  for (int r = 0; r < L; ++r) {
    double v = bb[r];
    for (int k = 0; k < r; ++k) v -= A[r][k] * bb[k];
    bb[r] = v / A[r][r];
  }
  for (int r = L - 1; r >= 0; --r) {
    double v = bb[r];
    for (int k = r + 1; k < L; ++k) v -= A[k][r] * bb[k];
    bb[r] = v / A[r][r];
  }
  return true;
}

__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }

template <int W>
__device__ __forceinline__ ff::F2 shfl_ff(ff::F2 a, int src) {
  return {__shfl_sync(0xffffffffu, a.hi, src, W), __shfl_sync(0xffffffffu, a.lo, src, W)};
}

// Shared memory of one subject's system.
struct PaceSys {
  double A[SC_LMAX][SC_LMAX + 1];  // Phi'Phi, both triangles
  double b[SC_LMAX];               // Phi'Y^C, then the scores
  double x[SC_LMAX];
  float2 low[SC_LMAX][SC_LMAX + 1];
};

// (A + diag(prior)) a = b for 32 / RL subjects of a warp, RL lanes each (lane r owns row r),
// the scores left in sys->b.  A chain of dependent FP64 operations is what one thread's
// FP64 Cholesky would wait on (~135 ns each here), so the factor is taken in float-float of
// the system scaled to a unit-size diagonal by powers of two, and the solution refined once
// with the FP64 residual: its error is the square of the float-float solve's, below FP64's
// own for what passes the test on the correction (2^-25 of the solution).  What does not
// pass (near-singular, not finite, extreme scales) is solved by one lane in FP64.
template <int RL>
__device__ void pace_solve(PaceSys* sys, const double* __restrict__ prior, int L, bool active,
                           int* err) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, r = lane % RL;
  const unsigned seg = (RL == 32 ? full : ((1u << RL) - 1u)) << (lane / RL * RL);
  const bool in = r < L;
  const bool valid = prior[SC_LMAX] != 0.0;
  if (active && in) sys->A[r][r] += prior[r];
  __syncwarp();
  const double dg = in && active ? sys->A[r][r] : 1.0, br = in && active ? sys->b[r] : 0.0;
  const int ex = ((__double2hiint(dg) >> 20) & 0x7ff) - 1023;
  bool fast = valid && dg > 0.0 && ex > -500 && ex < 500;
  const int sr = fast ? -(ex >> 1) : 0;  // 2^sr scales row and column r
  int eb = __double2hiint(br) & 0x7fffffff;
  for (int o = RL / 2; o > 0; o >>= 1) eb = max(eb, __shfl_xor_sync(full, eb, o, RL));
  eb = eb == 0 ? 0 : (eb >> 20) - 1023;
  if (eb < -500 || eb > 500) {
    fast = false;
    eb = 0;
  }
  ff::F2 a[RL];
#pragma unroll
  for (int c = 0; c < RL; ++c) {
    const int sc = __shfl_sync(full, sr, c, RL);
    a[c] = in && active && c < L ? split(sys->A[r][c] * pow2(sr + sc)) : ff::make(c == r ? 1.f : 0.f);
  }
  ff::F2 inv = ff::make(1.f);
#pragma unroll
  for (int j = 0; j < RL; ++j) {
    const ff::F2 p = shfl_ff<RL>(a[j], j);
    if (!(p.hi > 1e-7f)) fast = false;
    // 1 / sqrt(p): the FP32 value and one Newton step
    const float y0 = rsqrtf(fmaxf(p.hi, 1e-7f));
    const ff::F2 e = ff::add(ff::make(1.f), ff::neg(ff::mul(p, ff::two_prod(y0, y0))));
    const ff::F2 iv = ff::fast_two_sum(y0, 0.5f * y0 * e.hi);
    if (r == j) inv = iv;
    a[j] = ff::mul(a[j], iv);  // column j of the factor
    if (active) sys->low[r][j] = make_float2(a[j].hi, a[j].lo);
#pragma unroll
    for (int c = j + 1; c < RL; ++c) a[c] = ff::sub_mul(a[c], a[j], shfl_ff<RL>(a[j], c));
  }
  __syncwarp();
  auto solve = [&](ff::F2 v) {
    ff::F2 z = v;
#pragma unroll
    for (int k = 0; k < RL; ++k) {
      const ff::F2 xk = shfl_ff<RL>(ff::mul(z, inv), k);
      if (r == k) z = xk;
      if (r > k) z = ff::sub_mul(z, a[k], xk);
    }
#pragma unroll
    for (int k = RL - 1; k >= 0; --k) {
      const ff::F2 xk = shfl_ff<RL>(ff::mul(z, inv), k);
      if (r == k) z = xk;
      if (r < k) {
        const float2 lo = sys->low[k][r];
        z = ff::sub_mul(z, ff::F2{lo.x, lo.y}, xk);
      }
    }
    return z;
  };
  const ff::F2 x0 = solve(split(br * pow2(sr - eb)));
  if (active && in) sys->x[r] = ff::to_double(x0) * pow2(sr);
  __syncwarp();
  double r0 = br * pow2(-eb), r1 = 0.0;
  if (active && in) {
#pragma unroll
    for (int c = 0; c < RL; c += 2) {
      if (c < L) r0 = fma(-sys->A[r][c], sys->x[c], r0);
      if (c + 1 < L) r1 = fma(-sys->A[r][c + 1], sys->x[c + 1], r1);
    }
  }
  const ff::F2 dx = solve(split((r0 + r1) * pow2(sr)));
  float mx = fabsf(x0.hi), md = fabsf(dx.hi);
  if (!(mx < INFINITY) || !(md < INFINITY)) fast = false;
  for (int o = RL / 2; o > 0; o >>= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(full, mx, o, RL));
    md = fmaxf(md, __shfl_xor_sync(full, md, o, RL));
  }
  if (!(md <= 0x1p-25f * mx)) fast = false;
  const bool good = (__ballot_sync(full, !fast) & seg) == 0;
  if (active && good && in)
    sys->b[r] = (ff::to_double(x0) + ff::to_double(dx)) * pow2(sr) * pow2(eb);
  if (active && !good && r == 0) {
    if (!valid || !solve_serial(sys->A, sys->b, L)) {
      atomicExch(err, DERR_NUMERIC);
      for (int k = 0; k < L; ++k) sys->b[k] = __longlong_as_double(0x7ff8000000000000ll);
    }
  }
  __syncwarp();
}


// Scattered data (offs / t / y in FP64), mu2 (P) and phi2 (L x P) float-float: a warp per
// subject, its observations in chunks of 32 staged in shared memory, each lane a few of the
// NE + L sums.  LM: 8 or 16 >= L; the four subjects of a block are solved together, LM
// lanes each.  n = 20000, 5..20 points, 24 x 24, L = 8: 84 us; 617 us when one lane of each
// warp solved in FP64 and the chunks of 32 were always walked to their end.
template <int LM>
__global__ void __launch_bounds__(128)
    k_scores_pace(ScGrid g, int n, const void* __restrict__ y, const int64_t* __restrict__ offs,
                  const double* __restrict__ t, const float2* __restrict__ mu2,
                  const double* __restrict__ prior, const float2* __restrict__ phi2, int L,
                  double* __restrict__ scores, int* __restrict__ err) {
  constexpr int NS = (LM * (LM + 1) / 2 + LM + 31) / 32;  // sums per lane
  __shared__ float2 rows[4][32][LM + 1];                   // phi rows, then the residual
  __shared__ PaceSys sys[4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int NE = L * (L + 1) / 2;
  // Upper-triangle entries e = lane + 32 q (row-major) of Phi_i' Phi_i, then the L
  // entries of Phi_i' Y_i^C, held by this lane; er == LM: none
  int er[NS], ec[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    int r = 0, rem = lane + 32 * q;
    if (rem >= NE) {
      er[q] = rem - NE < L ? rem - NE : LM;
      ec[q] = LM;
      continue;
    }
    while (rem >= L - r) {
      rem -= L - r;
      ++r;
    }
    er[q] = r;
    ec[q] = r + rem;
  }
  const int i = blockIdx.x * 4 + warp;
  if (i < n) {
    Acc acc[NS];
    const long long j0 = offs[i], j1 = offs[i + 1];
    for (long long c0 = j0; c0 < j1; c0 += 32) {
      const long long j = c0 + lane;
      const int cnt = (int)(j1 - c0 < 32 ? j1 - c0 : 32);
      if (lane < cnt) {
        const int b = sc_bin(g, t + j * g.d);
        const float2 m = mu2[b];
        const ff::F2 yc = split(static_cast<const double*>(y)[j] - ((double)m.x + (double)m.y));
        for (int l = 0; l < L; ++l) rows[warp][lane][l] = phi2[(long long)l * g.P + b];
        rows[warp][lane][LM] = make_float2(yc.hi, yc.lo);
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < NS; ++q) {
        if (er[q] < LM) {
          for (int k = 0; k < cnt; ++k) {
            const float2 a = rows[warp][k][er[q]], c = rows[warp][k][ec[q]];
            acc[q].add_prod(ff::F2{a.x, a.y}, ff::F2{c.x, c.y});
          }
        }
      }
      __syncwarp();
    }
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      if (er[q] == LM) continue;
      const double v = acc[q].value();
      if (ec[q] == LM) {
        sys[warp].b[er[q]] = v;
      } else {
        sys[warp].A[er[q]][ec[q]] = v;
        sys[warp].A[ec[q]][er[q]] = v;
      }
    }
  }
  __syncthreads();
  constexpr int SPW = 32 / LM;  // subjects per solving warp
  if (warp < 4 / SPW) {
    const int sl = warp * SPW + lane / LM;
    pace_solve<LM>(&sys[sl], prior, L, blockIdx.x * 4 + sl < n, err);
  }
  __syncthreads();
  if (i < n && lane < L) scores[(long long)i * L + lane] = sys[warp].b[lane];
}

// ---------------------------------------------------------------------------
// gridded data
// ---------------------------------------------------------------------------
// (Phi_i'Phi_i)_ab = sum over nodes of mask_ip (phi_a phi_b)(p): a product of the 0/1 masks
// (n x P) with a P x NE table that no subject changes.  The table's entries are rounded to
// 54-bit fixed point relative to 2^(e_a + e_b) > max |phi_a| max |phi_b| and cut into five
// digits of 11 bits, which FP16 holds exactly; sums of up to PG_NODES digits are integers
// below 2^20, which the FP32 accumulators hold exactly, so the whole product is exact but for
// the table's rounding, 2^-54 of the bound a node.  That is closer than the float-float sums
// wherever a subject's mean phi_l^2 is above 2^-8 of the bound; the row of a function whose mean
// is smaller is summed in float-float (pace_rows).
constexpr int PG_DIG = 5;        // digits
constexpr int PG_BITS = 11;
constexpr int PG_FIX = 53;       // fixed-point bits
constexpr int PG_EBAD = 1000;    // exponent of a function that the digits cannot hold
constexpr int PG_EZERO = -1000;  // exponent of a function that is zero everywhere
constexpr int PG_COUNT = PG_BITS * (PG_DIG - 1);  // a leading digit of 1, as a fixed-point value

__host__ __device__ constexpr int pg_groups(int L) { return L * (L + 1) / 2 / 8 + 1; }

// The table in the order in which the product's B fragments are read: 64 nodes are four
// steps of 16; lane 4g + t of step j holds column g of the 8 and nodes 16 t + 4 j + {0..3},
// so that a lane's four steps of mask bytes are 16 consecutive ones.  Columns NE: a one
// (the subject's node count), beyond: zeros.  A block makes 64 nodes' worth, of the 64s from
// `first` on.
__global__ void __launch_bounds__(256)
    k_pace_table(int P, int first, int L, int nbx, const float* __restrict__ bmax,
                 const double* __restrict__ phi, uint2* __restrict__ table,
                 int* __restrict__ expo) {
  __shared__ double ph[SC_LMAX][64];
  __shared__ int ex[SC_LMAX];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int NE = L * (L + 1) / 2, ng = pg_groups(L), p0 = (first + blockIdx.x) * 64;
  for (int l = warp; l < L; l += 8) {
    float top = 0.f;
    for (int b = lane; b < nbx; b += 32) top = fmaxf(top, bmax[(long long)l * nbx + b]);
    for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    if (lane == 0) {
      int e = PG_EZERO;
      if (top > 0.f) {
        e = top < INFINITY ? ilogbf(top) + 1 : PG_EBAD;
        if (e < -60 || e > 60) e = PG_EBAD;
      }
      ex[l] = e;
      if (blockIdx.x == 0) expo[l] = e;
    }
  }
  for (int e = threadIdx.x; e < L * 64; e += 256) {
    const int l = e >> 6, p = p0 + (e & 63);
    ph[l][e & 63] = p < P ? phi[(long long)l * P + p] : 0.0;
  }
  __syncthreads();
  for (int it = threadIdx.x; it < ng * 128; it += 256) {
    const int t = it & 3, gcol = (it >> 2) & 7, j = (it >> 5) & 3, grp = it >> 7;
    const int e = grp * 8 + gcol;
    int a = 0, rem = e;
    while (a < L && rem >= L - a) {
      rem -= L - a;
      ++a;
    }
    const int b = a + rem;
    unsigned short dig[PG_DIG][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int q = 16 * t + 4 * j + i;
      long long x = 0;
      if (e < NE) {
        const int ea = ex[a], eb = ex[b];
        if (ea > PG_EZERO && ea < PG_EBAD && eb > PG_EZERO && eb < PG_EBAD)
          x = __double2ll_rn(ph[a][q] * ph[b][q] * pow2(PG_FIX - ea - eb));
      } else if (e == NE && p0 + q < P) {
        x = 1ll << PG_COUNT;
      }
#pragma unroll
      for (int d = PG_DIG - 1; d >= 0; --d) {
        const int half = 1 << (PG_BITS - 1);
        const int dv = d ? (int)((x + half) & (2 * half - 1)) - half : (int)x;
        x = (x - dv) >> PG_BITS;
        dig[d][i] = __half_as_ushort(__int2half_rn(dv));
      }
    }
#pragma unroll
    for (int d = 0; d < PG_DIG; ++d)
      table[((size_t)(blockIdx.x * 4 + j) * ng * PG_DIG + grp * PG_DIG + d) * 32 + gcol * 4 + t] =
          make_uint2(dig[d][0] | (unsigned)dig[d][1] << 16, dig[d][2] | (unsigned)dig[d][3] << 16);
  }
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const unsigned (&a)[4], uint2 b) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// 0xff for each nonzero byte of the mask's 16 nodes p..p+15 of a row (NULL: all observed),
// zero beyond the grid
__device__ __forceinline__ uint4 mask16(const uint8_t* __restrict__ row, int p, int P, int vec) {
  uint4 w = make_uint4(0, 0, 0, 0);
  if (vec && p < P) {
    if (row) {
      w = *reinterpret_cast<const uint4*>(row + p);
      w.x = __vcmpne4(w.x, 0);
      w.y = __vcmpne4(w.y, 0);
      w.z = __vcmpne4(w.z, 0);
      w.w = __vcmpne4(w.w, 0);
    } else {
      w = make_uint4(~0u, ~0u, ~0u, ~0u);
    }
  } else if (!vec) {
    unsigned u[4] = {0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (p + i < P && (!row || row[p + i])) u[i >> 2] |= 0xffu << (8 * (i & 3));
    w = make_uint4(u[0], u[1], u[2], u[3]);
  }
  return w;
}

// out[(split * nb + i) * 8 ng + e]: the fixed-point sums over the split's nodes.  A warp takes
// 16 subjects (its A fragments come straight from the mask's bytes) and GP groups of 8
// columns; blockIdx: x 128 subjects, y a split of `per` x 64 nodes, from the 64s `first` on, of
// which the table holds `have`, z GP groups.  1.5 GFLOP
// at n = 1000, P = 4096, L = 8 in 10 us: bound by the table's reads from L1/L2, so the simpler
// warp-level products are as good as tcgen05's here.
template <int GP>
__global__ void __launch_bounds__(256)
    k_pace_gram(int nb, int i0, int P, int first, int have, int ng, int per,
                const uint8_t* __restrict__ mask, const uint2* __restrict__ table,
                long long* __restrict__ out, int vec) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gr = lane >> 2, t = lane & 3;
  const int ra = blockIdx.x * 128 + warp * 16 + gr, rb = ra + 8;
  if (ra - gr >= nb) return;
  const int g0 = blockIdx.z * GP, gn = min(GP, ng - g0);
  const int k0 = first + blockIdx.y * per, k1 = min(first + have, k0 + per);
  float acc[GP][PG_DIG][4] = {};
  const bool oka = ra < nb, okb = rb < nb;
  const uint8_t* rowa = mask ? mask + (size_t)(i0 + (oka ? ra : 0)) * P : nullptr;
  const uint8_t* rowb = mask ? mask + (size_t)(i0 + (okb ? rb : 0)) * P : nullptr;
  // the fragments of the next 16 nodes are loaded while these are multiplied (the loads took
  // 0.95 of the time when each was waited for)
  const uint2* tb = table + ((size_t)(k0 - first) * 4 * ng + g0) * PG_DIG * 32 + lane;
  const size_t tstep = (size_t)ng * PG_DIG * 32;
  uint2 b[2][GP * PG_DIG];
  auto fetch = [&](uint2 (&f)[GP * PG_DIG]) {
#pragma unroll
    for (int q = 0; q < GP; ++q)
      if (q < gn) {
#pragma unroll
        for (int d = 0; d < PG_DIG; ++d) f[q * PG_DIG + d] = tb[(q * PG_DIG + d) * 32];
      }
    tb += tstep;
  };
  auto masks = [&](const uint8_t* row, bool ok, int k) {
    return ok && k < k1 ? mask16(row, k * 64 + t * 16, P, vec) : make_uint4(0, 0, 0, 0);
  };
  uint4 wa = masks(rowa, oka, k0), wb = masks(rowb, okb, k0);
  if (k0 < k1) fetch(b[0]);
  for (int k = k0; k < k1; ++k) {
    const unsigned ua[4] = {wa.x, wa.y, wa.z, wa.w}, ub[4] = {wb.x, wb.y, wb.z, wb.w};
    wa = masks(rowa, oka, k + 1);
    wb = masks(rowb, okb, k + 1);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const unsigned one = 0x3c003c00u;  // 1.0 where the byte is set
      const unsigned a[4] = {__byte_perm(ua[j], 0, 0x1404) & one, __byte_perm(ub[j], 0, 0x1404) & one,
                             __byte_perm(ua[j], 0, 0x3424) & one, __byte_perm(ub[j], 0, 0x3424) & one};
      if (j < 3 || k + 1 < k1) fetch(b[(j + 1) & 1]);
#pragma unroll
      for (int q = 0; q < GP; ++q) {
        if (q < gn) {
#pragma unroll
          for (int d = 0; d < PG_DIG; ++d) mma_f16(acc[q][d], a, b[j & 1][q * PG_DIG + d]);
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < GP; ++q) {
    if (q >= gn) break;
    long long v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      v[c] = 0;
#pragma unroll
      for (int d = 0; d < PG_DIG; ++d) v[c] = v[c] * (1 << PG_BITS) + (int)acc[q][d][c];
    }
    const size_t o = ((size_t)blockIdx.y * nb + ra) * (8 * ng) + (g0 + q) * 8 + 2 * t;
    if (oka) *reinterpret_cast<longlong2*>(out + o) = make_longlong2(v[0], v[1]);
    if (okb)
      *reinterpret_cast<longlong2*>(out + o + (size_t)8 * 8 * ng) = make_longlong2(v[2], v[3]);
  }
}

// The table's bound does not hold for a function (exponent e) of a subject: its mean square is
// below 2^-8 of 2^(2e).  all, nodes: the upper 32 bits of the fixed-point sums of phi_l^2 (units
// of 2^(2e - PG_FIX)) and of the node count (2^-PG_COUNT), so that the exponents cancel.
__device__ __forceinline__ bool pace_small(long long all, long long nodes, int e) {
  return e > PG_EZERO && (e == PG_EBAD || all < 2 * nodes);
}
static_assert(PG_FIX - 8 == PG_COUNT + 1, "pace_small");
// Place of entry (a, b), a <= b, in the upper triangle.
__device__ __forceinline__ int pace_entry(int L, int a, int b) { return a * L - a * (a - 1) / 2 + b - a; }

// The warp's sums of NV lane values each: a halving butterfly (one add a sum instead of five),
// v[0] <- sum number `at` (returned; with NV < 32 several lanes hold the same one).
template <int NV>
__device__ __forceinline__ int warp_halve(ff::F2 (&v)[NV]) {
  const int lane = threadIdx.x & 31;
  int at = 0;
#pragma unroll
  for (int st = 0; st < 5; ++st) {
    const int o = 16 >> st, left = NV >> (st + 1);
    const bool up = lane & o;
    if (up) at += left;
#pragma unroll
    for (int k = 0; k < (left > 0 ? left : 1); ++k) {
      const ff::F2 give = up || left == 0 ? v[k] : v[k + left];
      const ff::F2 keep = up && left > 0 ? v[k + left] : v[k];
      v[k] = ff::add(keep, ff::F2{__shfl_xor_sync(0xffffffffu, give.hi, o),
                                  __shfl_xor_sync(0xffffffffu, give.lo, o)});
    }
  }
  return at;
}

// Rows `small` (a bit each) of one subject's Phi'Phi over a chunk's pn nodes, in float-float, by
// one warp; out: the chunk's entries of the subject.  Each row serves all its entries, so that a
// localised function costs L sums of the L (L + 1) / 2.
template <int LM, int CH>
__device__ __forceinline__ void pace_rows(unsigned small, const float2 (*ph)[CH], int pn,
                                          const uint8_t* __restrict__ row, int L, bool clean,
                                          float2* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  for (unsigned left = small; left; left &= left - 1) {
    const int l = __ffs(left) - 1;
    const unsigned done = small & ((1u << l) - 1u);  // entries of an earlier row
    Acc acc[LM];
#pragma unroll 2
    for (int c = lane; c < pn; c += 32) {
      const bool ok = !row || row[c];
      const float2 x = ph[l][c];
      const ff::F2 fl = ok ? ff::F2{x.x, x.y} : ff::make(0.f);
#pragma unroll
      for (int b = 0; b < LM; ++b) {
        if (b < L && !(done >> b & 1)) {
          const ff::F2 f{ph[b][c].x, ph[b][c].y};
          acc[b].add_prod(fl, clean || ok ? f : ff::make(0.f));
        }
      }
    }
    ff::F2 v[LM];
#pragma unroll
    for (int b = 0; b < LM; ++b) v[b] = ff::fast_two_sum(acc[b].s, acc[b].c);
    const int b = warp_halve<LM>(v);
    if (b < L && !(done >> b & 1))
      out[pace_entry(L, min(l, b), max(l, b))] = make_float2(v[0].hi, v[0].lo);
  }
}

// which[i]: the functions of subject i that the table does not hold, a bit each; a warp a subject.
// On grids of many splits, where k_pace_dots does not go through all of them in every block.
__global__ void __launch_bounds__(256)
    k_pace_check(int nb, int L, int nsplit, const int* __restrict__ expo,
                 const long long* __restrict__ gsum, unsigned* __restrict__ which) {
  const int s = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (s >= nb) return;
  const int NE = L * (L + 1) / 2, ng8 = 8 * pg_groups(L);
  long long nodes = 0;
  unsigned bits = 0;
  for (int f = -1; f < L; ++f) {
    const long long* g = gsum + (size_t)s * ng8 + (f < 0 ? NE : pace_entry(L, f, f));
    long long all = 0;
    for (int k = lane; k < nsplit; k += 32) all += g[(size_t)k * nb * ng8] >> 32;
    for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
    if (f < 0)
      nodes = all;
    else if (pace_small(all, nodes, expo[f]))
      bits |= 1u << f;
  }
  if (lane == 0) which[s] = bits;
}

// All rows at once, where most are wanted: rows A0..A1 - 1 of the triangle (at most NV entries,
// which is what the registers hold), ordered by column.
template <int LM, int CH, int A0, int A1, int NV>
__device__ __forceinline__ void pace_triangle(const float2 (*ph)[CH], int pn,
                                              const uint8_t* __restrict__ row, int L, bool clean,
                                              float2* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  if (A0 >= L) return;
  Acc acc[NV];
#pragma unroll 1
  for (int c = lane; c < pn; c += 32) {
    const bool ok = !row || row[c];
    ff::F2 fa[A1 - A0];
#pragma unroll
    for (int a = A0; a < A1; ++a) fa[a - A0] = ok ? ff::F2{ph[a][c].x, ph[a][c].y} : ff::make(0.f);
    int k = 0;
#pragma unroll
    for (int b = A0; b < LM; ++b) {
      if (b < L) {
        const ff::F2 f{ph[b][c].x, ph[b][c].y};
#pragma unroll
        for (int a = A0; a < A1; ++a)
          if (a <= b) acc[k + a - A0].add_prod(fa[a - A0], clean || ok ? f : ff::make(0.f));
      }
      k += (b < A1 ? b + 1 : A1) - A0;
    }
  }
  ff::F2 v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = ff::fast_two_sum(acc[k].s, acc[k].c);
  int k = warp_halve<NV>(v);
  for (int b = A0; b < L; ++b) {
    const int rows = (b < A1 ? b + 1 : A1) - A0;
    if (k < rows) {
      out[pace_entry(L, A0 + k, b)] = make_float2(v[0].hi, v[0].lo);
      break;
    }
    k -= rows;
  }
}

// Phi_i'Y_i^C over a chunk of nodes: the chunk's phi in shared memory, two subjects a warp,
// each lane both subjects' L compensated sums over every 32nd node (a phi value read serves
// both); the sums join in float-float (FP64 adds there would take longer than the sums
// themselves).  The same warp then forms the rows of its subjects' Phi'Phi that the table does
// not hold.  n = 1000, P = 4096, whole call: L = 8 83 us, 114 with one localised function, 197 with
// all of them; L = 13 142, 204 and 462 (all entries of such a subject one after the other, in the
// solving block: 604 and 742; all subjects' entries in float-float, before there was a table: 280
// and 404, which is still the better one where more than eight functions are all localised).
// blockIdx: x chunk, y 16 subjects; bpart[(chunk * nb + i) * L + l], rpart[(chunk * nb + i) * NE +
// entry].  This kernel, bound by its FP32 instructions, takes 38 us of the 83 and the systems 16
// (n = 1500, P = 1320, L = 13: 38 and 30); with phi from L2 and a block taking two whole subjects
// and their systems 53 and 131, one warp per 1/8 subject, forming Phi'Phi too, 269 and 293.
constexpr int PD_CHUNK = 512;  // nodes (256 with 16 functions: 155 us for L = 13)
template <int LM>
__global__ void __launch_bounds__(256, LM == 8 ? 4 : 2)
    k_pace_dots(int nb, int i0, int P, const void* __restrict__ y, int yprec,
                const uint8_t* __restrict__ mask, const float2* __restrict__ mu2,
                const float2* __restrict__ phi2, int L, const int* __restrict__ expo, int nsplit,
                const long long* __restrict__ gsum, const unsigned* __restrict__ checked,
                float2* __restrict__ bpart, float2* __restrict__ rpart) {
  constexpr int NV = 2 * LM, CH = PD_CHUNK;
  extern __shared__ __align__(16) float2 pds[];
  float2(*ph)[CH] = reinterpret_cast<float2(*)[CH]>(pds);
  float2* mus = pds + LM * CH;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int p0 = blockIdx.x * CH, pn = min(CH, P - p0);
  for (int e = tid; e < LM * CH; e += 256) {
    const int l = e / CH, c = e % CH;
    ph[l][c] = l < L && c < pn ? phi2[(long long)l * P + p0 + c] : make_float2(0.f, 0.f);
  }
  for (int c = tid; c < pn; c += 256) mus[c] = mu2[p0 + c];
  bool clean = true;  // no phi value that times a zero is not zero
  for (int l = 0; l < L; ++l) clean &= expo[l] != PG_EBAD;
  __syncthreads();
  const int s0 = blockIdx.y * 16 + warp * 2;
  if (s0 >= nb) return;
  const size_t row0 = (size_t)(i0 + s0) * P + p0, row1 = (size_t)(i0 + min(s0 + 1, nb - 1)) * P + p0;
  Acc acc[2][LM];
#pragma unroll 2
  for (int c = lane; c < pn; c += 32) {
    // unobserved responses are read and not used, so that no load waits for another
    const bool ok0 = !mask || mask[row0 + c], ok1 = s0 + 1 < nb && (!mask || mask[row1 + c]);
    const float2 m = mus[c];
    ff::F2 r0 = centred(y, yprec, row0 + c, ff::F2{m.x, m.y});
    ff::F2 r1 = centred(y, yprec, row1 + c, ff::F2{m.x, m.y});
    if (!ok0) r0 = ff::make(0.f);
    if (!ok1) r1 = ff::make(0.f);
#pragma unroll
    for (int l = 0; l < LM; ++l) {
      if (l < L) {
        const ff::F2 f{ph[l][c].x, ph[l][c].y};
        acc[0][l].add_prod(r0, clean || ok0 ? f : ff::make(0.f));
        acc[1][l].add_prod(r1, clean || ok1 ? f : ff::make(0.f));
      }
    }
  }
  ff::F2 v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k)
    v[k] = ff::fast_two_sum(acc[k / LM][k % LM].s, acc[k / LM][k % LM].c);
  const int at = warp_halve<NV>(v);
  const int sl = s0 + at / LM, l = at % LM;  // (with 16 sums two lanes hold the same one)
  if (sl < nb && l < L)
    bpart[((size_t)blockIdx.x * nb + sl) * L + l] = make_float2(v[0].hi, v[0].lo);
  // the table's bound: lanes 0..15 the functions of subject s0, 16..31 those of the next (from
  // k_pace_check where it ran)
  const int NE = L * (L + 1) / 2, ng8 = 8 * pg_groups(L), f = lane & 15, si = s0 + (lane >> 4);
  bool small = false;
  if (f < L && si < nb && checked) {
    small = checked[si] >> f & 1;
  } else if (f < L && si < nb) {
    const int e = expo[f];
    const long long* g = gsum + (size_t)si * ng8;
    const int ff = pace_entry(L, f, f);
    long long all = 0, nodes = 0;
#pragma unroll 8
    for (int k = 0; k < nsplit; ++k, g += (size_t)nb * ng8) {
      all += g[ff] >> 32;
      nodes += g[NE] >> 32;
    }
    small = pace_small(all, nodes, e);
  }
  const unsigned which = __ballot_sync(0xffffffffu, small);
  if (!which) return;
  for (int h = 0; h < 2; ++h) {
    const unsigned rows = which >> (16 * h) & 0xffffu;
    const uint8_t* row = mask ? mask + (h ? row1 : row0) : nullptr;
    float2* out = rpart + ((size_t)blockIdx.x * nb + s0 + h) * NE;
    if (2 * __popc(rows) <= L) {
      pace_rows<LM, CH>(rows, ph, pn, row, L, clean, out);
    } else if constexpr (LM == 8) {
      pace_triangle<LM, CH, 0, 2, 16>(ph, pn, row, L, clean, out);
      pace_triangle<LM, CH, 2, 4, 16>(ph, pn, row, L, clean, out);
      pace_triangle<LM, CH, 4, 8, 16>(ph, pn, row, L, clean, out);
    } else {
      pace_triangle<LM, CH, 0, 2, 32>(ph, pn, row, L, clean, out);
      pace_triangle<LM, CH, 2, 4, 32>(ph, pn, row, L, clean, out);
      pace_triangle<LM, CH, 4, 6, 32>(ph, pn, row, L, clean, out);
      pace_triangle<LM, CH, 6, 9, 32>(ph, pn, row, L, clean, out);
      pace_triangle<LM, CH, 9, 16, 32>(ph, pn, row, L, clean, out);
    }
  }
}

// The systems of 32 / LM subjects: the sums of the node splits and chunks (the chunks' rows where
// the table's bound does not hold), and the solves.
template <int LM>
__global__ void __launch_bounds__(128)
    k_pace_final(int nb, int i0, const double* __restrict__ prior, int L, int nsplit, int nchunk,
                 const int* __restrict__ expo, const long long* __restrict__ gsum,
                 const float2* __restrict__ bpart, const float2* __restrict__ rpart,
                 double* __restrict__ scores, int* __restrict__ err) {
  constexpr int SUB = 32 / LM;
  __shared__ PaceSys sys[SUB];
  __shared__ long long top[SUB][SC_LMAX + 1];  // upper halves of the diagonal's sums, the count's
  __shared__ unsigned small[SUB];              // a bit per row from rpart
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NE = L * (L + 1) / 2, ng8 = 8 * pg_groups(L);
  const int s0 = blockIdx.x * SUB;
  if (tid < SUB) small[tid] = 0;
  for (int it = tid; it < SUB * (NE + 1 + L); it += 128) {
    const int sl = it / (NE + 1 + L), e = it - sl * (NE + 1 + L);
    if (s0 + sl >= nb) continue;
    if (e > NE) {
      const int l = e - NE - 1;
      double b0 = 0.0, b1 = 0.0;
      for (int k = 0; k < nchunk; ++k) {
        const float2 v = bpart[((size_t)k * nb + s0 + sl) * L + l];
        b0 += (double)v.x;
        b1 += (double)v.y;
      }
      sys[sl].b[l] = b0 + b1;
      continue;
    }
    long long hi = 0, lo = 0;  // of the splits' fixed-point sums
#pragma unroll 4
    for (int k = 0; k < nsplit; ++k) {
      const long long v = gsum[((size_t)k * nb + s0 + sl) * ng8 + e];
      hi += v >> 32;
      lo += v & 0xffffffffll;
    }
    if (e == NE) {
      top[sl][SC_LMAX] = hi;
      continue;
    }
    int a = 0, rem = e;
    while (rem >= L - a) {
      rem -= L - a;
      ++a;
    }
    const int b = a + rem, es = expo[a] + expo[b];
    if (a == b) top[sl][a] = hi;
    const double v = fma((double)hi, 4294967296.0, (double)lo);
    const double ge = es > -200 && es < 200 ? v * pow2(es - PG_FIX) : 0.0;
    sys[sl].A[a][b] = ge;
    sys[sl].A[b][a] = ge;
  }
  __syncthreads();
  bool any = false;
  if (tid < SUB * L) {
    const int sl = tid / L, l = tid - sl * L;
    any = s0 + sl < nb && pace_small(top[sl][l], top[sl][SC_LMAX], expo[l]);
    if (any) atomicOr(&small[sl], 1u << l);
  }
  if (__syncthreads_or(any)) {
    for (int it = tid; it < SUB * NE; it += 128) {
      const int sl = it / NE, e = it - sl * NE;
      int a = 0, rem = e;
      while (rem >= L - a) {
        rem -= L - a;
        ++a;
      }
      if (!((small[sl] >> a | small[sl] >> (a + rem)) & 1)) continue;
      double t = 0.0;
      for (int k = 0; k < nchunk; ++k) {
        const float2 v = rpart[((size_t)k * nb + s0 + sl) * NE + e];
        t += (double)v.x + (double)v.y;
      }
      sys[sl].A[a][a + rem] = t;
      sys[sl].A[a + rem][a] = t;
    }
    __syncthreads();
  }
  if (warp == 0) {
    const int sl = lane / LM;
    pace_solve<LM>(&sys[sl], prior, L, s0 + sl < nb, err);
    for (int e = lane; e < SUB * L; e += 32)
      if (s0 + e / L < nb) scores[(long long)(i0 + s0) * L + e] = sys[e / L].b[e % L];
  }
}

// A_il = dV sum_p mask (Y_ip - mu_p) phi_l(p): one block of 8 warps per subject,
// compensated per-thread sums joined in FP64 (shuffles, then the warps in order).
template <int LM>
__global__ void __launch_bounds__(256)
    k_scores_integral(int n, int P, const void* __restrict__ y, int yprec,
                      const uint8_t* __restrict__ mask, const float2* __restrict__ mu2,
                      const float2* __restrict__ phi2, int L, double dv,
                      double* __restrict__ scores) {
  __shared__ double wsum[8][LM];
  const int i = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long row = (long long)i * P;
  Acc acc[LM];
  for (int p = threadIdx.x; p < P; p += 256) {
    if (mask && !mask[row + p]) continue;
    const float2 m = mu2[p];
    const ff::F2 r = centred(y, yprec, row + p, ff::F2{m.x, m.y});
#pragma unroll
    for (int l = 0; l < LM; ++l) {
      if (l < L) {
        const float2 f = phi2[(long long)l * P + p];
        acc[l].add_prod(r, ff::F2{f.x, f.y});
      }
    }
  }
#pragma unroll
  for (int l = 0; l < LM; ++l) {
    double v = acc[l].value();
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) wsum[warp][l] = v;
  }
  __syncthreads();
  if (threadIdx.x < L) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += wsum[w][threadIdx.x];
    scores[(long long)i * L + threadIdx.x] = v * dv;
  }
}

// X_i(p) = mu_p + sum_l A_il phi_l(p), compensated, rounded once to FP32.  A
// thread keeps node p's mu and phi in registers and walks RC_SUB subjects whose
// scores were split into shared memory once per block.
constexpr int RC_SUB = 16;
template <int LM>
__global__ void __launch_bounds__(256)
    k_reconstruct(int n, int P, const float2* __restrict__ mu2, const float2* __restrict__ phi2,
                  int L, const double* __restrict__ scores, float* __restrict__ xhat) {
  __shared__ float2 a2[RC_SUB][LM];
  const int i0 = blockIdx.y * RC_SUB;
  for (int e = threadIdx.x; e < RC_SUB * LM; e += blockDim.x) {
    const int ii = e / LM, l = e - ii * LM;
    ff::F2 v = ff::make(0.f);
    if (i0 + ii < n && l < L) v = split(scores[(long long)(i0 + ii) * L + l]);
    a2[ii][l] = make_float2(v.hi, v.lo);
  }
  __syncthreads();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const float2 m = mu2[p];
  float2 f[LM];
#pragma unroll
  for (int l = 0; l < LM; ++l) f[l] = l < L ? phi2[(long long)l * P + p] : make_float2(0.f, 0.f);
  for (int ii = 0; ii < RC_SUB && i0 + ii < n; ++ii) {
    Acc acc;
    acc.s = m.x;
    acc.c = m.y;
#pragma unroll
    for (int l = 0; l < LM; ++l)
      if (l < L) acc.add_prod(ff::F2{a2[ii][l].x, a2[ii][l].y}, ff::F2{f[l].x, f[l].y});
    xhat[(long long)(i0 + ii) * P + p] = acc.s + acc.c;
  }
}

// Per-block partial sums of (xhat - x)^2 (compensated per thread, pairwise tree
// per block).
constexpr int MS_THREADS = 256;
__global__ void __launch_bounds__(MS_THREADS)
    k_mise_partial(long long ne, const float* __restrict__ xhat, const void* __restrict__ x,
                   int xprec, double* __restrict__ part) {
  __shared__ double red[MS_THREADS];
  Acc acc;
  for (long long e = blockIdx.x * (long long)MS_THREADS + threadIdx.x; e < ne;
       e += (long long)gridDim.x * MS_THREADS) {
    ff::F2 d;
    if (xprec == FPCA_F64)
      d = split((double)xhat[e] - static_cast<const double*>(x)[e]);
    else
      d = ff::two_sum(xhat[e], -static_cast<const float*>(x)[e]);
    acc.add_prod(d, d);
  }
  red[threadIdx.x] = acc.value();
  __syncthreads();
  for (int h = MS_THREADS / 2; h >= 1; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// out = scale * (sum of the nb partials), fixed pairwise tree in one block.
__global__ void __launch_bounds__(MS_THREADS)
    k_mise_final(int nb, const double* __restrict__ part, double scale, double* __restrict__ out) {
  __shared__ double red[MS_THREADS];
  double v = 0.0;
  for (int b = threadIdx.x; b < nb; b += MS_THREADS) v += part[b];
  red[threadIdx.x] = v;
  __syncthreads();
  for (int h = MS_THREADS / 2; h >= 1; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0] * scale;
}

ScGrid sc_grid(const fpca_grid* g) {
  ScGrid s{};
  s.d = g->d;
  s.P = 1;
  for (int k = 0; k < 3; ++k) {
    s.m[k] = k < g->d ? g->m[k] : 1;
    if (k < g->d) s.P *= g->m[k];
  }
  return s;
}

bool sc_valid_grid(fpca_ctx* ctx, const fpca_grid* g) {
  if (!g || g->d < 1 || g->d > 3) {
    fpca_fail(ctx, FPCA_E_INVALID_ARG, "grid.d must be 1..3");
    return false;
  }
  for (int k = 0; k < g->d; ++k)
    if (g->m[k] < 1) {
      fpca_fail(ctx, FPCA_E_INVALID_ARG, "grid.m[%d] must be positive", k);
      return false;
    }
  return true;
}

bool sc_valid(fpca_ctx* ctx, const fpca_grid* g, int L) {
  if (!sc_valid_grid(ctx, g)) return false;
  if (L < 1 || L > SC_LMAX) {
    fpca_fail(ctx, FPCA_E_INVALID_ARG, "L must be 1..%d", SC_LMAX);
    return false;
  }
  return true;
}

// Gridded data in batches of subjects and slabs of nodes: the scratch of fpca_scores_pace does
// not grow with n, and on the largest grids it stays below that of the functions' copies.
constexpr int PG_BATCH = 16384;   // subjects x splits ...
constexpr int PG_MOST = 65536;    // ... and beyond 512 splits, where 128 subjects are more
constexpr int PG_SLAB = 4096;     // 64s of nodes whose table is held at a time (2^18 nodes)
static_assert(PG_SLAB % 8 == 0, "whole splits in a slab");
// Splits up to which k_pace_dots tests the table's bound itself (32 splits, 128 x 128 nodes,
// n = 500: 132 us, 138 with k_pace_check; 512 splits, n = 100: 920 and 716).
constexpr int PG_INLINE = 64;

struct ScWork {
  float2 *mu2, *phi2;  // mu (P) and the first L eigenfunctions (L x P) as float-float
  double* prior;       // see k_split_ff
  // PACE of gridded data
  float* bmax;         // L x nbx block maxima of |phi|
  int* expo;           // L exponents
  uint2* table;
  long long* gsum;
  unsigned* which;        // k_pace_check
  float2 *bpart, *rpart;  // partial Phi'Y^C and rows of Phi'Phi of the node chunks
  const double* phi;
  int nbx, nsplit, per, batch, nchunk;
};

// mu and phi in float-float; with `grid` also what PACE of gridded data works with.  The other
// calls take none of that: at 2^20 nodes and L = 16 it is 2.4 GB beside their 0.14.
fpca_status sc_split(fpca_ctx* ctx, int P, int L, const double* mu, const double* evecs, ScWork* w,
                     const double* lam = nullptr, const double* sigma2 = nullptr, bool grid = false) {
  const int n64 = (P + 63) / 64, ng = pg_groups(L);
  *w = ScWork{};
  w->phi = evecs;
  w->nbx = std::min((P + 255) / 256, grid ? 64 : 4096);
  // 256 nodes a split, 512 on grids that make plenty of them: digit sums stay below 2^20,
  // fixed-point sums below 2^63
  w->per = n64 <= 64 ? 4 : 8;
  w->nsplit = (n64 + w->per - 1) / w->per;
  w->batch = w->nsplit <= PG_MOST / 128 ? std::max(128, PG_BATCH / w->nsplit / 128 * 128)
                                        : std::max(16, PG_MOST / w->nsplit / 16 * 16);
  w->nchunk = (P + PD_CHUNK - 1) / PD_CHUNK;
  const size_t nt = (size_t)std::min(n64, PG_SLAB) * 4 * ng * PG_DIG * 32;
  const size_t ns = (size_t)w->nsplit * w->batch * 8 * ng;
  const size_t nc = (size_t)w->nchunk * w->batch;
  const size_t nr = (size_t)L * (L + 1) / 2;
  size_t need = WsCarve::round(sizeof(float2) * P) + WsCarve::round(sizeof(float2) * (size_t)L * P) + 512;
  if (grid)
    need += WsCarve::round(sizeof(float) * L * w->nbx) + 512 + WsCarve::round(sizeof(uint2) * nt) +
            WsCarve::round(sizeof(long long) * ns) + WsCarve::round(sizeof(unsigned) * w->batch) +
            WsCarve::round(sizeof(float2) * nc * L) +
            WsCarve::round(sizeof(float2) * nc * nr);
  void* ws = fpca_workspace(ctx, need);
  if (!ws) return fpca_fail(ctx, FPCA_E_OOM, "workspace (%zu bytes)", need);
  WsCarve c(ws);
  w->mu2 = c.take<float2>(P);
  w->phi2 = c.take<float2>((size_t)L * P);
  w->prior = c.take<double>(SC_LMAX + 1);
  if (grid) {
    w->bmax = c.take<float>((size_t)L * w->nbx);
    w->expo = c.take<int>(SC_LMAX);
    w->table = c.take<uint2>(nt);
    w->gsum = c.take<long long>(ns);
    w->which = c.take<unsigned>(w->batch);
    w->bpart = c.take<float2>(nc * L);
    w->rpart = c.take<float2>(nc * nr);
  }
  k_split_ff<<<dim3(w->nbx, L + 1), 256, 0, ctx->stream>>>(P, mu, evecs, w->mu2, w->phi2, w->bmax, L,
                                                                lam, sigma2, w->prior);
  FPCA_LAUNCHED(ctx, "split_ff");
  return FPCA_OK;
}

fpca_status pace_dense(fpca_ctx* ctx, const fpca_data* data, int P, int L, const ScWork& w,
                       double* scores) {
  const int n64 = (P + 63) / 64, ng = pg_groups(L), gp = ng <= 2 ? 2 : 5;
  // 16 mask bytes at once where rows are whole multiples of them
  const int vec = P % 16 == 0 && (reinterpret_cast<uintptr_t>(data->mask) & 15) == 0;
  auto gram = gp == 2 ? k_pace_gram<2> : k_pace_gram<5>;
  for (int i0 = 0; i0 < data->n; i0 += w.batch) {
    const int nb = std::min(w.batch, data->n - i0);
    for (int first = 0; first < n64; first += PG_SLAB) {  // (whole splits)
      const int have = std::min(PG_SLAB, n64 - first);
      if (i0 == 0 || n64 > PG_SLAB) {
        k_pace_table<<<have, 256, 0, ctx->stream>>>(P, first, L, w.nbx, w.bmax, w.phi, w.table, w.expo);
        FPCA_LAUNCHED(ctx, "pace_table");
      }
      gram<<<dim3((nb + 127) / 128, (have + w.per - 1) / w.per, (ng + gp - 1) / gp), 256, 0,
             ctx->stream>>>(nb, i0, P, first, have, ng, w.per, data->mask, w.table,
                            w.gsum + (size_t)(first / w.per) * nb * 8 * ng, vec);
      FPCA_LAUNCHED(ctx, "pace_gram");
    }
    const bool check = w.nsplit > PG_INLINE;
    if (check) {
      k_pace_check<<<(nb + 7) / 8, 256, 0, ctx->stream>>>(nb, L, w.nsplit, w.expo, w.gsum, w.which);
      FPCA_LAUNCHED(ctx, "pace_check");
    }
    auto dots = L <= 8 ? k_pace_dots<8> : k_pace_dots<16>;
    const int dsm = (int)sizeof(float2) * PD_CHUNK * (L <= 8 ? 9 : 17);
    cudaFuncSetAttribute(dots, cudaFuncAttributeMaxDynamicSharedMemorySize, dsm);
    dots<<<dim3(w.nchunk, (nb + 15) / 16), 256, dsm, ctx->stream>>>(
        nb, i0, P, data->y, data->y_prec, data->mask, w.mu2, w.phi2, L, w.expo,
        w.nsplit, w.gsum, check ? w.which : nullptr, w.bpart, w.rpart);
    FPCA_LAUNCHED(ctx, "pace_dots");
    auto fin = L <= 8 ? k_pace_final<8> : k_pace_final<16>;
    const int sub = L <= 8 ? 4 : 2;
    fin<<<(nb + sub - 1) / sub, 128, 0, ctx->stream>>>(nb, i0, w.prior, L, w.nsplit, w.nchunk,
                                                      w.expo, w.gsum, w.bpart, w.rpart, scores,
                                                      ctx->d_err);
    FPCA_LAUNCHED(ctx, "scores_pace");
  }
  return FPCA_OK;
}

}  // namespace

extern "C" {

fpca_status fpca_scores_pace(fpca_ctx* ctx, const fpca_data* data, const fpca_grid* grid,
                             const double* mu, const double* evals, const double* evecs, int L,
                             const double* sigma2, double* scores) {
  if (!ctx) return FPCA_E_INVALID_ARG;
  fpca_prof_mark(ctx);
  if (!sc_valid(ctx, grid, L)) return FPCA_E_INVALID_ARG;
  if (!data || !mu || !evals || !evecs || !sigma2 || !scores)
    return fpca_fail(ctx, FPCA_E_INVALID_ARG,
                     "data, mu, evals, evecs, sigma2 and scores are required");
  if (data->n < 1 || !data->y) return fpca_fail(ctx, FPCA_E_INVALID_ARG, "data.n >= 1 and y");
  if (data->layout == FPCA_SPARSE && (!data->offs || !data->t))
    return fpca_fail(ctx, FPCA_E_INVALID_ARG, "scattered data need offs and t");
  const ScGrid g = sc_grid(grid);
  ScWork w;
  fpca_status s = sc_split(ctx, g.P, L, mu, evecs, &w, evals, sigma2, data->layout != FPCA_SPARSE);
  if (s != FPCA_OK) return s;
  if (data->layout == FPCA_SPARSE) {
    auto kern = L <= 8 ? k_scores_pace<8> : k_scores_pace<16>;
    kern<<<(data->n + 3) / 4, 128, 0, ctx->stream>>>(g, data->n, data->y, data->offs, data->t, w.mu2,
                                                     w.prior, w.phi2, L, scores, ctx->d_err);
    FPCA_LAUNCHED(ctx, "scores_pace");
    return FPCA_OK;
  }
  return pace_dense(ctx, data, g.P, L, w, scores);
}

fpca_status fpca_scores_integral(fpca_ctx* ctx, const fpca_data* data, const fpca_grid* grid,
                                 const double* mu, const double* evecs, int L, double* scores) {
  if (!ctx) return FPCA_E_INVALID_ARG;
  fpca_prof_mark(ctx);
  if (!sc_valid(ctx, grid, L)) return FPCA_E_INVALID_ARG;
  if (!data || !mu || !evecs || !scores)
    return fpca_fail(ctx, FPCA_E_INVALID_ARG, "data, mu, evecs and scores are required");
  if (data->layout != FPCA_DENSE || !data->y || data->n < 1)
    return fpca_fail(ctx, FPCA_E_INVALID_ARG, "scores by integration need gridded (dense) data");
  const ScGrid g = sc_grid(grid);
  ScWork w;
  fpca_status s = sc_split(ctx, g.P, L, mu, evecs, &w);
  if (s != FPCA_OK) return s;
  const double dv = 1.0 / (double)g.P;
  if (L <= 8)
    k_scores_integral<8><<<data->n, 256, 0, ctx->stream>>>(data->n, g.P, data->y, data->y_prec,
                                                           data->mask, w.mu2, w.phi2, L, dv, scores);
  else
    k_scores_integral<16><<<data->n, 256, 0, ctx->stream>>>(data->n, g.P, data->y, data->y_prec,
                                                            data->mask, w.mu2, w.phi2, L, dv, scores);
  FPCA_LAUNCHED(ctx, "scores_integral");
  return FPCA_OK;
}

fpca_status fpca_reconstruct(fpca_ctx* ctx, const fpca_grid* grid, const double* mu,
                             const double* evecs, int L, const double* scores, int n,
                             float* xhat) {
  if (!ctx) return FPCA_E_INVALID_ARG;
  fpca_prof_mark(ctx);
  if (!sc_valid(ctx, grid, L)) return FPCA_E_INVALID_ARG;
  if (!mu || !evecs || !scores || !xhat || n < 1)
    return fpca_fail(ctx, FPCA_E_INVALID_ARG, "mu, evecs, scores, xhat and n >= 1 are required");
  const int nsub = (n + RC_SUB - 1) / RC_SUB;
  if (nsub > 65535) return fpca_fail(ctx, FPCA_E_UNSUPPORTED, "more than 2^20 subjects per call");
  const ScGrid g = sc_grid(grid);
  ScWork w;
  fpca_status s = sc_split(ctx, g.P, L, mu, evecs, &w);
  if (s != FPCA_OK) return s;
  const dim3 grid2((g.P + 255) / 256, nsub);
  if (L <= 8)
    k_reconstruct<8><<<grid2, 256, 0, ctx->stream>>>(n, g.P, w.mu2, w.phi2, L, scores, xhat);
  else
    k_reconstruct<16><<<grid2, 256, 0, ctx->stream>>>(n, g.P, w.mu2, w.phi2, L, scores, xhat);
  FPCA_LAUNCHED(ctx, "reconstruct");
  return FPCA_OK;
}

fpca_status fpca_mise(fpca_ctx* ctx, const fpca_grid* grid, const float* xhat, const void* x,
                      int x_prec, int n, double* mise) {
  if (!ctx) return FPCA_E_INVALID_ARG;
  fpca_prof_mark(ctx);
  if (!sc_valid_grid(ctx, grid)) return FPCA_E_INVALID_ARG;
  if (!xhat || !x || !mise || n < 1)
    return fpca_fail(ctx, FPCA_E_INVALID_ARG, "xhat, x, mise and n >= 1 are required");
  if (x_prec != FPCA_F64 && x_prec != FPCA_F32)
    return fpca_fail(ctx, FPCA_E_INVALID_ARG, "x_prec must be FPCA_F64 or FPCA_F32");
  const ScGrid g = sc_grid(grid);
  const long long ne = (long long)n * g.P;
  const int nb = (int)std::min<long long>((ne + MS_THREADS - 1) / MS_THREADS,
                                          (long long)std::max(1, ctx->num_sms) * 8);
  double* part = static_cast<double*>(fpca_workspace(ctx, sizeof(double) * nb));
  if (!part) return fpca_fail(ctx, FPCA_E_OOM, "workspace");
  k_mise_partial<<<nb, MS_THREADS, 0, ctx->stream>>>(ne, xhat, x, x_prec, part);
  FPCA_LAUNCHED(ctx, "mise");
  k_mise_final<<<1, MS_THREADS, 0, ctx->stream>>>(nb, part, 1.0 / ((double)g.P * (double)n),
                                                  mise);
  FPCA_LAUNCHED(ctx, "mise");
  return FPCA_OK;
}

}  // extern "C"
