// One seed of the exhaustive search (Eq. codec, Sec. 3.1), split in two: what
// depends on the seed alone (the eliminated normal matrix) and what depends on
// the block (right-hand side, coefficients, exponent, error).  Both the
// exhaustive kernels and the screened search use these steps, so a (block,
// seed) pair gives the same bits wherever it is evaluated.
#pragma once

#include "seedq_internal.cuh"

namespace seedq {

// Power of two 2^e as a double (|e| well inside the normal range).
__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }

// The double equal to the integer +-mag * 2^e (mag < 2^63), built from bits.
__device__ __forceinline__ double exact_d(bool neg, unsigned long long mag, int e) {
  if (mag == 0) return 0.0;
  const int msb = 63 - __clzll((long long)mag);
  const unsigned long long mant = (msb <= 52 ? (mag << (52 - msb)) : (mag >> (msb - 52))) & ((1ull << 52) - 1);
  return __longlong_as_double((long long)(((unsigned long long)neg << 63) |
                                          ((unsigned long long)(1023 + msb + e) << 52) | mant));
}
__device__ __forceinline__ double i2d(long long v) {
  return exact_d(v < 0, (unsigned long long)(v < 0 ? -v : v), 0);
}
// |bits| of a double, as an integer whose order is the order of magnitudes.
__device__ __forceinline__ unsigned long long mag_bits(double d) {
  return (unsigned long long)__double_as_longlong(d) & 0x7fffffffffffffffull;
}
// d * 2^e for d normal or zero (exponent field shift).
__device__ __forceinline__ double scale2(double d, int e) {
  const long long b = __double_as_longlong(d);
  return (b & 0x7fffffffffffffffll) == 0 ? d : __longlong_as_double(b + ((long long)e << 52));
}

// All k round-half-even values of x_j * 2^e lie in [-8, 7], i.e. every
// x_j * 2^e lies in [-8.5, 7.5) (compared as bit patterns: exact).
template <int K>
__device__ __forceinline__ bool fits(const double (&x)[K], int e) {
  const unsigned long long lim_neg = (unsigned long long)__double_as_longlong(8.5);
  const unsigned long long lim_pos = (unsigned long long)__double_as_longlong(7.5);
  bool ok = true;
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const double v = scale2(x[j], e);
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    ok = ok && ((b >> 63) ? ((b & 0x7fffffffffffffffull) <= lim_neg) : (b < lim_pos));
  }
  return ok;
}

// The eliminated normal matrix of one seed: multipliers below the diagonal,
// the rows above it, the pivots with their reciprocal estimates, and the row
// exchanged at each step.  Stored as kDoubles 8-byte words per seed (a
// multiple of 16 bytes).
template <int K>
struct SeedFactor {
  static constexpr int kTri = K * (K - 1) / 2;
  static constexpr int kDoubles = (2 * kTri + 2 * K + 1 + 1) / 2 * 2;
  double f[kTri];     // multiplier of step c, row r: index tri(c, r)
  double up[kTri];    // A[c][q], q > c: index tri(c, q)
  DivRecip R[K];      // pivots
  uint32_t pr;        // row exchanged with row c at step c: bits [3c, 3c + 3)
  bool singular;
  static __host__ __device__ constexpr int tri(int c, int r) { return c * (2 * K - c - 1) / 2 + (r - c - 1); }

  __device__ __forceinline__ void store(double *row) const {
#pragma unroll
    for (int i = 0; i < kTri; ++i) {
      row[i] = f[i];
      row[kTri + i] = up[i];
    }
#pragma unroll
    for (int c = 0; c < K; ++c) {
      row[2 * kTri + c] = R[c].b;
      row[2 * kTri + K + c] = __longlong_as_double((long long)R[c].inv);
    }
    row[2 * kTri + 2 * K] = __longlong_as_double((long long)pr);
  }
  __device__ __forceinline__ void load(const double *row) {
    double v[kDoubles];
#pragma unroll
    for (int i = 0; i < kDoubles / 2; ++i) {
      const double2 d = __ldg(reinterpret_cast<const double2 *>(row) + i);
      v[2 * i] = d.x;
      v[2 * i + 1] = d.y;
    }
#pragma unroll
    for (int i = 0; i < kTri; ++i) {
      f[i] = v[i];
      up[i] = v[kTri + i];
    }
#pragma unroll
    for (int c = 0; c < K; ++c)
      R[c] = div_recip_from(v[2 * kTri + c], (uint64_t)__double_as_longlong(v[2 * kTri + K + c]));
    pr = (uint32_t)__double_as_longlong(v[2 * kTri + 2 * K]);
    singular = false;
  }
};

// U(s) scaled by 2^(S-1): the integers x - 2^(S-1).
template <int K>
__device__ __forceinline__ void seed_matrix(int S, uint64_t Q, int (&u)[8][K]) {
  const uint32_t mask = (1u << S) - 1u;
  const int h = 1 << (S - 1);
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < K; ++j) u[i][j] = (int)((uint32_t)(Q >> (i * K + j)) & mask) - h;
}

// Gaussian elimination with partial pivoting (first row of largest |pivot|) of
// the unscaled normal matrix (exact integers).  Divisions are exact IEEE
// quotients on the integer pipes (div_rn), one reciprocal estimate per pivot.
template <int K>
__device__ __forceinline__ void factor_seed(int S, const int (&u)[8][K], SeedFactor<K> &F) {
  double A[K][K];
#pragma unroll
  for (int p = 0; p < K; ++p)
#pragma unroll
    for (int q = p; q < K; ++q) {
      long long acc = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) acc += (long long)(u[i][p] * u[i][q]);
      A[p][q] = i2d(acc);
      A[q][p] = A[p][q];
    }
  // Pivot threshold of the unscaled matrix: 1e-12 * 2^(2S-2), exact.
  const unsigned long long thr = mag_bits(__dmul_rn(1e-12, pow2d(2 * S - 2)));
  F.singular = false;
  F.pr = 0;
#pragma unroll
  for (int c = 0; c < K; ++c) {
    int pr = c;
    unsigned long long pv = mag_bits(A[c][c]);
#pragma unroll
    for (int r = c + 1; r < K; ++r) {
      const unsigned long long v = mag_bits(A[r][c]);
      if (v > pv) {
        pv = v;
        pr = r;
      }
    }
    F.singular = F.singular || (pv < thr);
    F.pr |= (uint32_t)pr << (3 * c);
#pragma unroll
    for (int r = c + 1; r < K; ++r) {
      if (pr == r) {
#pragma unroll
        for (int q = c; q < K; ++q) {
          const double tmp = A[c][q];
          A[c][q] = A[r][q];
          A[r][q] = tmp;
        }
      }
    }
    F.R[c] = div_recip(A[c][c]);
#pragma unroll
    for (int r = c + 1; r < K; ++r) {
      const double f = div_rn(A[r][c], F.R[c]);
      F.f[F.tri(c, r)] = f;
#pragma unroll
      for (int q = c + 1; q < K; ++q) A[r][q] = __dsub_rn(A[r][q], __dmul_rn(f, A[c][q]));
    }
#pragma unroll
    for (int q = c + 1; q < K; ++q) F.up[F.tri(c, q)] = A[c][q];
  }
}

// The block's weights as integers m * 2^e (exact for floats).
struct BlockParts {
  double w[8];
  int32_t m[8];    // signed 24-bit mantissas
  uint32_t sh[8];  // e[i] - emin (0 for a zero weight)
  int emin;        // smallest exponent of a nonzero weight (0 when all are zero)
  bool exact;      // exponents within 11 of each other: see solve_block
  __device__ __forceinline__ explicit BlockParts(const float (&wf)[8]) {
    int emax = -(1 << 20), e[8];
    emin = 1 << 20;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      w[i] = (double)wf[i];
      const uint32_t fb = __float_as_uint(wf[i]);
      const int ef = (int)((fb >> 23) & 255u);
      const int mag = (int)((fb & 0x7fffffu) | (ef ? 0x800000u : 0u));
      m[i] = (fb >> 31) ? -mag : mag;
      e[i] = (ef ? ef : 1) - 150;
      if (mag) {
        emin = min(emin, e[i]);
        emax = max(emax, e[i]);
      }
    }
    exact = emax - emin <= 11;
    if (emin == (1 << 20)) emin = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) sh[i] = m[i] ? (uint32_t)(e[i] - emin) : 0u;
  }
};

// The right-hand side in the oracle's rounding order, for blocks whose
// exponents spread too far (rare, so kept out of line: the evaluation's code
// then fits the instruction cache better).
template <int K>
__device__ __noinline__ void rounded_rhs(int S, uint64_t Q, const float *wf, double *b) {
  const uint32_t mask = (1u << S) - 1u;
  const int h = 1 << (S - 1);
  for (int p = 0; p < K; ++p) {
    double r = 0.0;
    for (int i = 0; i < 8; ++i) {
      const int ui = (int)((uint32_t)(Q >> (i * K + p)) & mask) - h;
      const uint32_t fb = __float_as_uint(wf[i]);
      const int ef = (int)((fb >> 23) & 255u);
      const uint32_t m = (fb & 0x7fffffu) | (ef ? 0x800000u : 0u);
      // u * w is exact: built from the integer product of the mantissas.
      const double prod = exact_d((fb >> 31) != (uint32_t)(ui < 0),
                                  (unsigned long long)(ui < 0 ? -ui : ui) * m, (ef ? ef : 1) - 150);
      r = __dadd_rn(r, prod);
    }
    b[p] = r;
  }
}

// v * 2^e for |v| < 2^24 (exact): the bits of the float v, widened.
__device__ __forceinline__ double small_d(int v, int e) {
  const uint32_t f = __float_as_uint((float)v);
  const uint32_t hi = (f & 0x80000000u) | (((f & 0x7fffffffu) >> 3) + ((uint32_t)(896 + e) << 20));
  return v ? __hiloint2double((int)hi, (int)(f << 29)) : 0.0;
}

// Coefficients, exponent and quantized squared error of one block (weights wf,
// parts B) at one non-singular seed (its sequence prefix Q, matrix u, factor F).
template <int K>
__device__ __forceinline__ double solve_block(int S, uint64_t Q, const int (&u)[8][K], const SeedFactor<K> &F,
                                              const BlockParts &B, const float *wf, int &Eout, int (&t)[6]) {
  double b[K];
  if (B.exact) {
    // Right-hand side without rounding: when the weights' exponents lie within
    // 11 of each other, every product |u| * m (< 2^39) aligned to the smallest
    // exponent stays below 2^50, so every partial sum of the eight is an
    // integer below 2^53: each fp64 addition of the rounded sequence is then
    // exact, and its sum equals the integer sum.
#pragma unroll
    for (int p = 0; p < K; ++p) {
      long long acc = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) acc += (long long)(u[i][p] << B.sh[i]) * (long long)B.m[i];
      b[p] = exact_d(acc < 0, (unsigned long long)(acc < 0 ? -acc : acc), B.emin);
    }
  } else {
    double r[K];
    rounded_rhs<K>(S, Q, wf, r);
#pragma unroll
    for (int p = 0; p < K; ++p) b[p] = r[p];
  }
#pragma unroll
  for (int c = 0; c < K; ++c) {
    const int pr = (int)(F.pr >> (3 * c)) & 7;
#pragma unroll
    for (int r = c + 1; r < K; ++r) {
      if (pr == r) {
        const double tb = b[c];
        b[c] = b[r];
        b[r] = tb;
      }
    }
#pragma unroll
    for (int r = c + 1; r < K; ++r) b[r] = __dsub_rn(b[r], __dmul_rn(F.f[F.tri(c, r)], b[c]));
  }
  double x[K];
#pragma unroll
  for (int r = K - 1; r >= 0; --r) {
    double sacc = b[r];
#pragma unroll
    for (int q = r + 1; q < K; ++q) sacc = __dsub_rn(sacc, __dmul_rn(F.up[F.tri(r, q)], x[q]));
    x[r] = div_rn(sacc, F.R[r]);
  }
  // x = tstar * 2^-(S-1); the mantissa of t_j at exponent E is rint(x_j * 2^(S-1-E)).
  // fits() is monotone in E, so the smallest fitting E is found by stepping
  // from an estimate.
  unsigned long long xm = 0;
#pragma unroll
  for (int j = 0; j < K; ++j) xm = max(xm, mag_bits(x[j]));
  int E = xm ? ((int)(xm >> 52) - 1023) + (S - 1) - 2 : -8;
  E = E < -8 ? -8 : (E > 7 ? 7 : E);
  while (E > -8 && fits<K>(x, S - 1 - (E - 1))) --E;
  while (E < 7 && !fits<K>(x, S - 1 - E)) ++E;
#pragma unroll
  for (int j = 0; j < K; ++j) {
    double m = rint(scale2(x[j], S - 1 - E));
    m = m < -8.0 ? -8.0 : (m > 7.0 ? 7.0 : m);
    t[j] = (int)m;
  }
#pragma unroll
  for (int j = K; j < 6; ++j) t[j] = 0;
  // Quantized squared error, summed in i order.
  double err = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    int Ri = 0;
#pragma unroll
    for (int j = 0; j < K; ++j) Ri += u[i][j] * t[j];
    const double d = __dsub_rn(B.w[i], small_d(Ri, 1 - S + E));  // |Ri| <= 8 K 2^15 < 2^24
    err = __dadd_rn(err, __dmul_rn(d, d));
  }
  Eout = E;
  return err;
}

struct EncodeOut {
  uint32_t *seed;
  int8_t *E;
  int8_t *t;   // 6 per block
  double *err;
};

__device__ __forceinline__ void write_out(const EncodeOut &o, int64_t blk, double best, uint32_t bseed,
                                          int bE, const int (&bt)[6], int K) {
  o.seed[blk] = bseed;
  o.E[blk] = (int8_t)bE;
  for (int j = 0; j < 6; ++j) o.t[blk * 6 + j] = (int8_t)(j < K ? bt[j] : 0);
  if (o.err) o.err[blk] = best;
}

// The eight weights of block c of row r of W (R x C fp32, original column
// order).  Outlier columns are stored in FP16 and overwrite the decode (Sec.
// 3.5): the search sees them as zero, so their spike does not leak into the
// block-mates.
__device__ __forceinline__ void gather_block(const LayerArgs &p, const float *W, int64_t r, int c, float (&wv)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int col = __ldg(p.perm + 8 * c + i);
    bool outlier = false;
    for (int o = 0; o < p.n_out; ++o) outlier |= (p.out_cols[o] == col);
    wv[i] = outlier ? 0.f : __ldg(W + r * p.C + col);
  }
}

// Screened search (encode_screen.cu).  False when there was no memory for its
// scratch: nothing was launched, and the caller takes the exhaustive kernels.
// Any other failure is in *e.
bool screen_blocks(int S, int K, const float *w, int64_t nblocks, const EncodeOut &o, cudaStream_t st,
                   cudaError_t *e);
bool screen_layer(const seedq_layer *L, const float *W, const EncodeOut &o, cudaStream_t st, cudaError_t *e);

}  // namespace seedq
