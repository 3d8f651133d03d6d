// Screened seed search: the result of the exhaustive search (encode.cu), bit
// for bit, with the fp64 solve run only for the few seeds that can still win.
//
// The quantized error of a block w at seed s is at least the distance of w from
// span(U(s)), whatever the coefficients.  With an orthonormal basis of that
// span (K <= 3) or of its complement (K >= 4), fixed per seed, that distance
// is a few dot products of length 8: a matrix product of all seeds' vectors
// (depth 8) with all blocks, on the tensor cores.  A (block, seed) pair whose
// distance exceeds the best error found so far by more than the screening's
// own error bound cannot win and is dropped; the rest, 20 to 800 of the 65535
// at S = 16, are evaluated exactly as the exhaustive search would.
//
// The two per-seed parts, screening vectors and eliminated normal matrix, are
// written once per call by k_seed_tables.
//
// Work split of k_screen: a CTA takes a tile of 128 blocks (64 per half, when
// the tile has that many) and a range of seed groups; a warp holds its 64
// blocks as eight B fragments in registers and streams 16 seeds at a time
// through m16n8k8 FP16 products (one per screening vector, so a thread holds
// every vector's product of its (seed, block) pairs and forms the squared
// distance in place).  Survivors go to the warp's queue in shared memory and
// are evaluated 32 at a time, one per lane.  Tiles that are too few for the
// GPU are split by seed range; the last CTA of a tile to arrive combines the
// ranges.  The winner (smallest error, then smallest seed) does not depend on
// the order of evaluation.
//
// What bounds it: at (16, 3) the latency of the product chain (16 warps per
// SM; issue active 44% of cycles, tensor pipe 45%) ahead of the fp64 pipe (the
// evaluations, 28 a block); at K >= 5 the evaluations (200 to 1000 a block).
// Measured on one GB300 against the exhaustive kernels (every pair solved):
// 32768 blocks at (16, 3) 446 -> 0.84 ms (39 M blocks/s; the 2.1 G pairs'
// products alone are 0.17 ms of tensor time), 32768 blocks of a 4-bit layer
// (rungs (12, 3) to (16, 6)) 455 -> 1.2 ms, 1000 blocks at (16, 6) 82 -> 0.85
// ms.  Tried: TF32 fragments 5% to 15% slower (twice the registers and table
// bytes at the same 11 significant bits); three CTAs per SM 4% slower (80
// registers spill the evaluation); one launch per rung 1.9x slower on a layer.
//
// Screening error: vectors and weights (scaled into [-2, 2]) are rounded to FP16 (2^-11 each), so a
// dot product is off by at most kDotErr |w|: 2^-10, and a tenth of that for the
// float32 sums and the vectors' own error (float32 where a seed's columns lose
// at most a factor of 16 to one another, which leaves under 2e-5; fp64 up to
// 2^20; beyond that a seed is never dropped).  Captured energy (K <= 3) is then
// off by 2 sqrt(K) kDotErr |w|^2 + K kDotErr^2 |w|^2, the distance (K >= 4) by
// sqrt(8 - K) kDotErr |w|.
#include <cuda_fp16.h>

#include "encode_core.cuh"

namespace seedq {
namespace {

constexpr int kTile = 128;              // blocks per tile
constexpr int kScreenWarps = 8;
constexpr int kScreenThreads = 32 * kScreenWarps;
constexpr int kTableThreads = 64;
constexpr int kQueue = 31 + 16 * 64;    // survivors a warp can hold: a remainder and a whole group's
constexpr int kSampleGroups = 8;        // groups a warp ranks for the first threshold (4: 1% to 4% slower)
constexpr double kDotErr = 1.1 / 1024.0;
constexpr float kFloatLoss = 256.f;     // float32 vectors up to a growth of 16 (in length)

// Screening vectors per seed: the span's K, or the complement's 8 - K.
template <int K>
struct Screen {
  static constexpr bool kSpan = K <= 3;
  static constexpr int m = kSpan ? K : 8 - K;
};
__host__ __device__ constexpr double sqrt_int(int n) {  // n in 2..4
  return n == 2 ? 1.4142135623730951 : n == 3 ? 1.7320508075688774 : 2.0;
}

// Per-rung tables in device memory.
struct SeedTables {
  uint2 *frag;      // (group * m + v) * 32 + lane: A fragment of vector v of 16 seeds
  uint32_t *mask;   // per group: bits 0-15 never drop, bits 16-31 never evaluate
  double *rows;     // 2^S x SeedFactor<K>::kDoubles
  uint64_t *jump;   // 512 LFSR jump table entries
};

struct Part {
  uint64_t err;  // bits
  uint32_t seed;
};

// One rung of a call.
struct RungJob {
  int S, K;
  uint32_t taps;
  int cta0;                // first block of its table launch
  SeedTables tab;
  const int64_t *first;    // layer: blocks of this rung before row r (R + 1 entries), else nullptr
};

struct ScreenArgs {
  RungJob job[kMaxJ];      // in rising order of rung
  int njobs;
  EncodeOut out;
  const float *w;          // list: nblocks x 8
  int64_t nblocks;
  const float *W;          // layer: R x C
  Part *part;              // records of split tiles: kTile per item
  uint64_t *gbest;         // per block of a split tile: smallest error so far (bits; kNoBest: none)
  uint32_t *arrive;        // per split tile: splits finished (0 at the start of a call)
  uint32_t *next;          // next item (0 at the start of a call)
  uint32_t *wide;          // seeds (| rung << 16) whose vectors need fp64
  uint32_t *nwide;         // their number (0 at the start of a call)
  int64_t max_split;       // split items (and tiles) the records hold
};

// A block's error before any is known: the largest pattern of one repeated
// byte that is a finite double, so one memset writes it.
constexpr uint64_t kNoBest = 0x7f7f7f7f7f7f7f7full;

__device__ __forceinline__ uint32_t pack_half(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ int64_t block_count(const ScreenArgs &a, int j, int64_t R) {
  return a.job[j].first ? a.job[j].first[R] : a.nblocks;
}

// ------------------------------------------------------------- seed tables

// First 64 sequence bits from a seed, by the window recurrence.
__device__ __forceinline__ uint64_t lfsr_prefix(int S, uint32_t taps, uint32_t seed) {
  uint64_t q = seed;
  for (int t = S; t < 64; ++t) q |= (uint64_t)(__popcll((q >> (t - S)) & taps) & 1) << t;
  return q;
}

// Householder QR of V (8 x K); x = Q e_(first + v) for the m screening vectors
// goes to the A fragments of m16n8k8: columns 2q, 2q + 1 of row g, then of row
// g + 8 (lane 4g + q).  Returns the squared product of each column's length over
// what is left of it once the earlier columns are projected out, the factor by
// which rounding errors can grow (infinite when a column vanishes).
template <int K, typename T>
__device__ __forceinline__ T screening_vectors(T (&V)[8][K], uint2 *frag, uint32_t s) {
  T beta[K], loss = T(1);
#pragma unroll
  for (int j = 0; j < K; ++j) {
    // Reflections keep lengths: the column's own is that of all 8 rows now.
    T n0 = T(0), sg = T(0);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      n0 += V[i][j] * V[i][j];
      if (i >= j) sg += V[i][j] * V[i][j];
    }
    loss *= sg > T(0) ? n0 / sg : T(INFINITY);
    const T al = V[j][j] > T(0) ? -sqrt(sg) : sqrt(sg);
    V[j][j] -= al;
    T vv = T(0);
#pragma unroll
    for (int i = j; i < 8; ++i) vv += V[i][j] * V[i][j];
    beta[j] = vv > T(0) ? T(2) / vv : T(0);
#pragma unroll
    for (int k = j + 1; k < K; ++k) {
      T d = T(0);
#pragma unroll
      for (int i = j; i < 8; ++i) d += V[i][j] * V[i][k];
      d *= beta[j];
#pragma unroll
      for (int i = j; i < 8; ++i) V[i][k] -= d * V[i][j];
    }
  }
  const int r = s & 15, g = r & 7, hi = r >> 3;
#pragma unroll
  for (int v = 0; v < Screen<K>::m; ++v) {
    T x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = i == (Screen<K>::kSpan ? v : K + v) ? T(1) : T(0);
#pragma unroll
    for (int j = K - 1; j >= 0; --j) {
      T d = T(0);
#pragma unroll
      for (int i = j; i < 8; ++i) d += V[i][j] * x[i];
      d *= beta[j];
#pragma unroll
      for (int i = j; i < 8; ++i) x[i] -= d * V[i][j];
    }
#pragma unroll
    for (int i = 0; i < 8; i += 2)
      reinterpret_cast<uint32_t *>(frag + (size_t)((s >> 4) * Screen<K>::m + v) * 32 + g * 4 + i / 2)[hi] =
          pack_half((float)x[i], (float)x[i + 1]);
  }
  return loss;
}

// One thread per seed.  Neighbouring columns of U overlap in all but one bit
// per entry: 2 u_j - u_(j-1) is a vector of signs (times 2^(S-1), less one
// bit), and the columns are close to dependent when two of these agree up to
// sign (one pair in 128).  So the span's basis is taken over u_0 and the sign
// vectors, one of an agreeing pair replaced by the pair's difference (exact
// integers); a float32 QR of those is then good for all but 3% of the seeds
// at K = 6 and fewer below.  The rest go to a list for the fp64 kernel.
template <int K>
__device__ __forceinline__ void seed_table(const RungJob &a, int j, uint32_t s, uint32_t *wide, uint32_t *nwide) {
  const int S = a.S;
  for (uint32_t v = s; v < 512; v += 1u << S) a.tab.jump[v] = jump_table_entry(S, a.taps, v);
  int u[8][K];
  seed_matrix<K>(S, lfsr_prefix(S, a.taps, s), u);
  bool never;
  {
    SeedFactor<K> F;
    factor_seed<K>(S, u, F);
    never = F.singular || s == 0;
    F.store(a.tab.rows + (size_t)s * SeedFactor<K>::kDoubles);
  }
#pragma unroll
  for (int k = K - 1; k > 0; --k)
#pragma unroll
    for (int i = 0; i < 8; ++i) u[i][k] = 2 * u[i][k] - u[i][k - 1];
  // Sign patterns of u_1..u_(K-1) (all entries nonzero: they are near +-2^(S-1)).
  uint32_t sg[K];
#pragma unroll
  for (int k = 1; k < K; ++k) {
    sg[k] = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) sg[k] |= (uint32_t)(u[i][k] < 0) << i;
  }
#pragma unroll
  for (int k = 2; k < K; ++k) {
    bool done = false;
#pragma unroll
    for (int p = 1; p < k; ++p) {
      const uint32_t d = sg[k] ^ sg[p];
      if (!done && (d == 0 || d == 255u)) {
        // u_p may itself be a difference by now; then it stays as it is.
        bool sign_vector = true;
#pragma unroll
        for (int i = 0; i < 8; ++i) sign_vector = sign_vector && abs(u[i][p]) > 1;
        if (sign_vector) {
#pragma unroll
          for (int i = 0; i < 8; ++i) u[i][k] += d == 0 ? -u[i][p] : u[i][p];
          done = true;
        }
      }
    }
  }
  float V[8][K];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int k = 0; k < K; ++k) V[i][k] = (float)u[i][k];
  const float loss = screening_vectors<K, float>(V, a.tab.frag, s);
  if (!never && !(loss < kFloatLoss)) wide[atomicAdd(nwide, 1u)] = s | ((uint32_t)j << 16);
  const int lane = threadIdx.x & 31;
  const uint32_t nv = __ballot_sync(0xffffffffu, never);
  if ((lane & 15) == 0) a.tab.mask[s >> 4] = ((nv >> (lane & 16)) & 0xffffu) << 16;
}

// The tables of every rung of a call in one launch (kMaxK: the largest K
// among them, which sets the registers).
template <int kMaxK>
__global__ void __launch_bounds__(kTableThreads) k_seed_tables(const __grid_constant__ ScreenArgs a, int64_t R) {
  int j = 0;
  while (j + 1 < a.njobs && (int)blockIdx.x >= a.job[j + 1].cta0) ++j;
  if (block_count(a, j, R) == 0) return;
  const RungJob &J = a.job[j];
  const uint32_t s = (blockIdx.x - J.cta0) * kTableThreads + threadIdx.x;  // 2^S is a multiple of kTableThreads
  switch (J.K) {
    case 2: seed_table<2>(J, j, s, a.wide, a.nwide); break;
    case 3: if constexpr (kMaxK >= 3) seed_table<3>(J, j, s, a.wide, a.nwide); break;
    case 4: if constexpr (kMaxK >= 4) seed_table<4>(J, j, s, a.wide, a.nwide); break;
    case 5: if constexpr (kMaxK >= 5) seed_table<5>(J, j, s, a.wide, a.nwide); break;
    default: if constexpr (kMaxK >= 6) seed_table<6>(J, j, s, a.wide, a.nwide); break;
  }
}

template <int K>
__device__ __forceinline__ void seed_table_wide(const RungJob &a, uint32_t s) {
  int u[8][K];
  seed_matrix<K>(a.S, lfsr_prefix(a.S, a.taps, s), u);
  double V[8][K];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int k = 0; k < K; ++k) V[i][k] = (double)u[i][k];
  const double loss = screening_vectors<K, double>(V, a.tab.frag, s);
  // 2^20 in length is 2^40 here; fp64 then still leaves 2^-32.
  if (!(loss < 1099511627776.0)) atomicOr(a.tab.mask + (s >> 4), 1u << (s & 15));
}

__global__ void __launch_bounds__(kTableThreads) k_seed_tables_wide(const __grid_constant__ ScreenArgs a) {
  const uint32_t n = *a.nwide;
  for (uint32_t i = blockIdx.x * kTableThreads + threadIdx.x; i < n; i += gridDim.x * kTableThreads) {
    const RungJob &J = a.job[a.wide[i] >> 16];
    const uint32_t s = a.wide[i] & 0xffffu;
    switch (J.K) {
      case 2: seed_table_wide<2>(J, s); break;
      case 3: seed_table_wide<3>(J, s); break;
      case 4: seed_table_wide<4>(J, s); break;
      case 5: seed_table_wide<5>(J, s); break;
      default: seed_table_wide<6>(J, s); break;
    }
  }
}

// ------------------------------------------------------------------ search

struct __align__(16) TileState {
  float w[kTile][8];
  uint32_t bfrag[2][8][32];              // per half: B fragments of eight 8-block columns
  uint64_t jump[512];
  double sc[kTile];                      // scale of an error to the scaled block
  uint64_t best[kScreenWarps][64];       // per warp: smallest error of its blocks (bits)
  uint32_t bseed[kScreenWarps][64];      // and its seed (0: none yet)
  uint32_t queue[kScreenWarps][kQueue];  // survivors: seed | block << 16
  int qn[kScreenWarps];                  // their number
  float n2[kTile];                       // |w|^2 of the scaled block
  float ntau[kTile];                     // minus the threshold (see threshold())
  int64_t blk[kTile];                    // output index, -1 past the end
  uint8_t live[kTile];
  uint64_t *gbest;                       // the tile's shared errors when it is split, else nullptr
  uint64_t seen[kTile];                  // the shared error the threshold already allows for
  int64_t item;
  int last;
  // The call's plan: per rung, its blocks, splits per tile, first item, first
  // split item and first split tile.
  int64_t count[kMaxJ], item0[kMaxJ + 1], sitem0[kMaxJ], stile0[kMaxJ];
  int splits[kMaxJ];
};

// Errors are never negative, so they order as their bit patterns.
constexpr uint64_t kInfBits = 0x7ff0000000000000ull;

// A pair survives when (captured energy) + ntau >= 0 for K <= 3, when
// (distance^2) + ntau < 0 for K >= 4.  best: bits of the smallest error so far;
// sc scales it to the scaled block, whose |w|^2 is n2.  The small factors cover
// the float32 roundings here, in n2 (each below 1e-6) and in the sums.
template <int K>
__device__ __forceinline__ float threshold(float n2, uint64_t best, double sc) {
  constexpr double rm = sqrt_int(Screen<K>::m), e = kDotErr;
  const float bs = __double2float_ru(__longlong_as_double((long long)best) * sc);
  if (Screen<K>::kSpan) return bs * (1.f + 4e-6f) + n2 * (float)(2.0 * rm * e + Screen<K>::m * e * e - 1.0 + 4e-6);
  const float d = sqrtf(bs) + (float)(rm * e) * sqrtf(n2);
  return -(d * d) * (1.f + 8e-6f);
}
// The value no pair survives (blocks past the end or not finite).
template <int K>
__device__ __forceinline__ float threshold_none() {
  return Screen<K>::kSpan ? -INFINITY : INFINITY;
}
template <int K>
__device__ __forceinline__ bool tighter(float a, float b) {
  return Screen<K>::kSpan ? a < b : a > b;
}

// Exact evaluation of one (block, seed) pair.
template <int K>
__device__ __forceinline__ double evaluate(const TileState &T, int S, const double *rows, int b, uint32_t seed,
                                           int &E, int (&t)[6]) {
  const uint64_t Q = T.jump[seed & 255u] ^ T.jump[256 + (seed >> 8)];
  int u[8][K];
  seed_matrix<K>(S, Q, u);
  SeedFactor<K> F;
  F.load(rows + (size_t)seed * SeedFactor<K>::kDoubles);
  float w[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) w[i] = T.w[b][i];
  return solve_block<K>(S, Q, u, F, BlockParts(w), T.w[b], E, t);
}

// Evaluate n queue entries starting at q0 (n <= 32), one per lane, and lower
// the warp's best errors and the blocks' thresholds.
template <int K>
__device__ __noinline__ void drain(TileState &T, int S, const double *rows, int q0, int n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t ent = lane < n ? T.queue[warp][q0 + lane] : 0u;
  const uint32_t seed = ent & 0xffffu;
  const int b = (int)(ent >> 16);
  uint64_t err = 0;
  if (lane < n) {
    int E, t[6];
    err = (uint64_t)__double_as_longlong(evaluate<K>(T, S, rows, b, seed, E, t));
  }
  // One lane per block at a time: the lowest of those that still improve it.
  bool cand = lane < n;
  while (true) {
    const uint64_t be = T.best[warp][b & 63];
    cand = cand && (err < be || (err == be && seed < T.bseed[warp][b & 63]));
    const unsigned m = __ballot_sync(0xffffffffu, cand);
    if (!m) break;
    if (cand) {
      const unsigned same = __match_any_sync(m, b);
      if (lane == __ffs(same) - 1) {
        T.best[warp][b & 63] = err;
        T.bseed[warp][b & 63] = seed;
        // Other warps may lower the same threshold at the same time: each
        // value written is a valid one, so whichever stays is valid.
        const float nt = threshold<K>(T.n2[b], err, T.sc[b]);
        if (tighter<K>(nt, T.ntau[b])) T.ntau[b] = nt;
        if (T.gbest) atomicMin((unsigned long long *)T.gbest + b, (unsigned long long)err);
        cand = false;
      }
    }
    __syncwarp();
  }
  __syncwarp();
}

template <int K>
__device__ __noinline__ void write_winner(const TileState &T, int S, const double *rows, const EncodeOut &o, int b,
                                          uint64_t err, uint32_t seed) {
  int E = 0, t[6] = {0, 0, 0, 0, 0, 0};
  if (seed) evaluate<K>(T, S, rows, b, seed, E, t);
  write_out(o, T.blk[b], __longlong_as_double((long long)err), seed, E, t, K);
}

template <int M>
__device__ __forceinline__ void load_group(const SeedTables &t, int g, int lane, uint2 (&A)[M]) {
#pragma unroll
  for (int v = 0; v < M; ++v) A[v] = __ldg(t.frag + ((size_t)g * M + v) * 32 + lane);
}

__device__ __forceinline__ void mma_f16(float (&d)[4], uint2 A, uint32_t b) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%7,%7,%7,%7};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(A.x), "r"(A.y), "r"(b), "f"(0.f));
}

// Squared length of the m products of 16 seeds x 8 blocks on top of init
// (packed pairs of neighbouring blocks).
template <int M>
__device__ __forceinline__ void group_tile(const uint2 (&A)[M], uint32_t b, uint64_t init, float (&c)[4]) {
  uint64_t lo = init, hi = init;
#pragma unroll
  for (int v = 0; v < M; ++v) {
    float d[4];
    mma_f16(d, A[v], b);
    const uint64_t p = f2_pack(d[0], d[1]), q = f2_pack(d[2], d[3]);
    lo = f2_fma(p, p, lo);
    hi = f2_fma(q, q, hi);
  }
  const float2 l = f2_unpack(lo), h = f2_unpack(hi);
  c[0] = l.x;
  c[1] = l.y;
  c[2] = h.x;
  c[3] = h.y;
}

// Modeled time of a group of 16 seeds against a tile, by K: its products and,
// for K >= 5, the survivors they leave.
__host__ __device__ constexpr int group_cost(int K) { return K == 2 ? 2 : K == 3 ? 3 : K == 4 ? 5 : K == 5 ? 10 : 30; }

// The call's items: every rung's tiles, split by seed range so that an item is
// about a third of a CTA's share, in order of falling rung (the costliest
// first) and, within a rung, split by split: a later range of a tile then
// starts from the errors the earlier ones found.
__device__ void plan_items(TileState &T, const ScreenArgs &a, int64_t R, int64_t ctas) {
  int64_t total = 0, all = 0;
  for (int j = 0; j < a.njobs; ++j) {
    T.count[j] = block_count(a, j, R);
    all += (T.count[j] + kTile - 1) / kTile;
    total += (T.count[j] + kTile - 1) / kTile * (((1 << a.job[j].S) >> 4) * group_cost(a.job[j].K));
  }
  const int64_t target = total / (3 * ctas) + 1;
  int64_t item = 0, sitem = 0, stile = 0;
  for (int i = 0; i < a.njobs; ++i) {
    const int j = a.njobs - 1 - i;
    const int groups = (1 << a.job[j].S) >> 4;
    const int64_t tiles = (T.count[j] + kTile - 1) / kTile, cost = (int64_t)groups * group_cost(a.job[j].K);
    int64_t s = (cost + target / 2) / target;
    // With tiles for half the CTAs or more, ranges of 16 groups at least; with
    // fewer, of eight, with one for sixteen of four (of two at S = 8), where the
    // evaluations of weights that no seed stands out for (too small or too large
    // for any exponent) would keep few CTAs busy: 4000 blocks of standard deviation
    // 1e-4 at (8, 4) 1903 -> 369 us, 1000 at (10, 4) 1760 -> 579; of 0.02 (8, 4) x
    // 1000 128 -> 103, (10, 2) x 4000 87 -> 90.
    int most = groups / 16;
    if (2 * all <= ctas) {
      const int fine = groups == 16 ? groups / 2 : 16 * all <= ctas ? groups / 4 : groups / 8;
      most = fine < 64 ? fine : most > 64 ? most : 64;
    }
    s = s > most ? most : s;
    if (s < 1 || sitem + tiles * s > a.max_split) s = 1;  // the records are that many
    T.splits[i] = (int)s;
    T.item0[i] = item;
    T.sitem0[i] = sitem;
    T.stile0[i] = stile;
    item += tiles * s;
    if (s > 1) {
      sitem += tiles * s;
      stile += tiles;
    }
  }
  T.item0[a.njobs] = item;
}

template <int K, bool kLayer>
__device__ __noinline__ void run_item(TileState &T, const ScreenArgs &a, const LayerArgs &p, int i, int64_t local) {
  constexpr int M = Screen<K>::m;
  constexpr bool kSpan = Screen<K>::kSpan;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, g = lane >> 2, q = lane & 3;
  const int j = a.njobs - 1 - i;
  const RungJob &J = a.job[j];
  const int S = J.S, groups = (1 << S) >> 4, splits = T.splits[i];
  const int64_t total = T.count[j], tiles = (total + kTile - 1) / kTile;
  const int split = (int)(local / tiles);
  const int64_t tile = local - split * tiles;
  const int64_t stile = T.stile0[i] + tile;
  const int g0 = (int)((int64_t)groups * split / splits), g1 = (int)((int64_t)groups * (split + 1) / splits);
  const int nv = (int)min((int64_t)kTile, total - tile * kTile);
  for (int v = t; v < 512; v += kScreenThreads) T.jump[v] = J.tab.jump[v];
  // Load the tile.
  if (t < kTile) {
    const int64_t n = tile * kTile + t;
    float w[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    int64_t blk = -1;
    if (t < nv) {
      if constexpr (kLayer) {
        int64_t lo = 0, hi = p.R - 1;  // row holding the rung's block n
        while (lo < hi) {
          const int64_t mid = (lo + hi + 1) >> 1;
          if (J.first[mid] <= n) lo = mid;
          else hi = mid - 1;
        }
        const int c = (j > 0 ? p.brk[lo * (p.J - 1) + j - 1] : 0) + (int)(n - J.first[lo]);
        gather_block(p, a.W, lo, c, w);
        blk = lo * p.nb + c;
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = __ldg(a.w + n * 8 + e);
        blk = n;
      }
    }
    // Scaled by a power of two so that the largest weight lies in [1, 2).
    float mx = 0.f;
    bool fin = true;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      T.w[t][e] = w[e];
      fin = fin && isfinite(w[e]);
      mx = fmaxf(mx, fabsf(w[e]));
    }
    // A zero block is decided below (every error is zero); a block with a NaN
    // or an infinity has no error below infinity at any seed.
    const bool live = t < nv && fin && mx > 0.f;
    const int ex = live ? ilogbf(mx) : 0;
    float ws[8], n2 = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      ws[e] = live ? scalbnf(w[e], -ex) : 0.f;
      n2 = fmaf(ws[e], ws[e], n2);
    }
    // B fragment of m16n8k8: rows 2q, 2q + 1 of column g (lane 4g + q).
#pragma unroll
    for (int e = 0; e < 4; ++e)
      T.bfrag[t >> 6][(t >> 3) & 7][(t & 7) * 4 + e] = pack_half(ws[2 * e], ws[2 * e + 1]);
    const double sc = pow2d(-2 * ex);
    float nt = threshold_none<K>();
    uint64_t gb = kNoBest;
    if (live) {
      nt = kSpan ? INFINITY : -INFINITY;
      if (splits > 1) gb = __ldcg(a.gbest + stile * kTile + t);
      if (gb < kNoBest) nt = threshold<K>(n2, gb, sc);
    }
    T.seen[t] = gb;
    T.blk[t] = blk;
    T.live[t] = live;
    T.n2[t] = n2;
    T.sc[t] = sc;
    T.ntau[t] = nt;
  }
  for (int k = t; k < kScreenWarps * 64; k += kScreenThreads) {
    T.best[k >> 6][k & 63] = kInfBits;
    T.bseed[k >> 6][k & 63] = 0u;
  }
  if (t < kScreenWarps) T.qn[t] = 0;
  if (t == 0) T.gbest = splits > 1 ? a.gbest + stile * kTile : nullptr;
  __syncthreads();
  // Two halves of 64 blocks with four seed streams each, or one with eight.
  const bool wide = nv > 64;
  const int half = wide ? warp >> 2 : 0, hb = half * 64;
  const int stream = wide ? warp & 3 : warp, streams = wide ? 4 : 8;
  const int nt = min(8, (nv - hb + 7) >> 3);
  if (stream == 0) {
    // Zero blocks: the smallest seed that is not skipped.
    for (int k = lane; k < 64 && hb + k < nv; k += 32) {
      bool zero = true;
#pragma unroll
      for (int e = 0; e < 8; ++e) zero = zero && T.w[hb + k][e] == 0.f;
      if (!zero) continue;
      uint32_t s = 0;
      for (int gi = 0; gi < groups && s == 0; ++gi) {
        const uint32_t ok = ~(J.tab.mask[gi] >> 16) & 0xffffu;
        if (ok) s = gi * 16 + __ffs(ok) - 1;
      }
      if (s) {
        T.best[warp][k] = 0ull;
        T.bseed[warp][k] = s;
      }
    }
  }
  // First thresholds, unless an earlier range left one for every block: rank
  // the warp's first groups and evaluate each block's closest seed.
  bool known = true;
  for (int k = lane; k < 64; k += 32) known = known && !(T.live[hb + k] && isinf(T.ntau[hb + k]));
  if (!__all_sync(0xffffffffu, known)) {
    float sv[16];
    uint32_t ss[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      sv[k] = -1.f;
      ss[k] = 0u;
    }
    for (int k = 0; k < kSampleGroups; ++k) {
      const int gi = g0 + stream + k * streams;
      if (gi >= g1) break;
      uint2 A[M];
      load_group<M>(J.tab, gi, lane, A);
      const uint32_t skip = J.tab.mask[gi] | (J.tab.mask[gi] >> 16);
#pragma unroll
      for (int n = 0; n < 8; ++n) {
        float c[4];
        group_tile<M>(A, T.bfrag[half][n][lane], 0ull, c);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int r = g + 8 * (e >> 1), k2 = 2 * n + (e & 1);
          // Larger is closer; |w|^2 < 32 after scaling.
          const float score = (skip >> r & 1u) ? -1.f : kSpan ? c[e] : 64.f - c[e];
          if (score > sv[k2]) {
            sv[k2] = score;
            ss[k2] = gi * 16 + r;
          }
        }
      }
    }
    int qn = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
#pragma unroll
      for (int off = 4; off < 32; off <<= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, sv[k], off);
        const uint32_t os = __shfl_xor_sync(0xffffffffu, ss[k], off);
        if (ov > sv[k] || (ov == sv[k] && os < ss[k])) {
          sv[k] = ov;
          ss[k] = os;
        }
      }
      const int b = hb + (k >> 1) * 8 + 2 * q + (k & 1);
      const bool has = lane < 4 && (k >> 1) < nt && T.live[b] && sv[k] >= 0.f;
      const unsigned m = __ballot_sync(0xffffffffu, has);
      if (has) T.queue[warp][qn + __popc(m & ((1u << lane) - 1u))] = ss[k] | ((uint32_t)b << 16);
      qn += __popc(m);
    }
    __syncwarp();
    while (qn > 0) {
      const int n = min(qn, 32);
      qn -= n;
      drain<K>(T, S, J.tab.rows, qn, n);
    }
  }
  __syncthreads();
  // Every seed of the range.  The products run without a call in between (so
  // that the fragments stay in registers) until 32 survivors wait.
  int gi = g0 + stream;
  while (gi < g1) {
    uint32_t B[8];
#pragma unroll
    for (int n = 0; n < 8; ++n) B[n] = T.bfrag[half][n][lane];
    // One group against the warp's blocks, four 8-block columns at a time:
    // their products overlap, and survivors (rare) are looked for once.
    auto step = [&](const uint2(&A)[M], int gr, uint32_t mask) {
#pragma unroll
      for (int n0 = 0; n0 < 8; n0 += 4) {
        if (n0 >= nt) break;
        float c[4][4];
        int any = kSpan ? -1 : 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint64_t init = *reinterpret_cast<const volatile uint64_t *>(&T.ntau[hb + (n0 + k) * 8 + 2 * q]);
          group_tile<M>(A, B[n0 + k], init, c[k]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (kSpan) any &= __float_as_int(c[k][e]);
            else any |= __float_as_int(c[k][e]);
          }
        if ((kSpan ? any >= 0 : any < 0) || (mask & 0xffffu)) {
          // The 16 sign bits, pair (k, e) at bit 15 - 4k - e; rows g at e < 2,
          // g + 8 above.
          uint32_t sv = 0;
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) sv = __funnelshift_l((uint32_t)__float_as_int(c[k][e]), sv, 1);
          if (kSpan) sv ^= 0xffffu;
          const uint32_t mr = mask >> g;
          sv |= ((mr & 1u) ? 0xccccu : 0u) | ((mr >> 8 & 1u) ? 0x3333u : 0u);
          sv &= ~(((mr >> 16 & 1u) ? 0xccccu : 0u) | ((mr >> 24 & 1u) ? 0x3333u : 0u));
          while (sv) {
            const int at = 15 - (31 - __clz((int)sv)), e = at & 3;
            sv &= ~(0x8000u >> at);
            const int b = hb + (n0 + (at >> 2)) * 8 + 2 * q + (e & 1);
            if (T.live[b])
              T.queue[warp][atomicAdd(&T.qn[warp], 1)] = (uint32_t)(gr * 16 + g + 8 * (e >> 1)) | ((uint32_t)b << 16);
          }
        }
      }
      __syncwarp();
      return *reinterpret_cast<const volatile int *>(&T.qn[warp]);
    };
    // The next group's fragments load while one is in hand.
    uint2 A0[M], A1[M];
    uint32_t m0 = __ldg(J.tab.mask + gi), m1;
    load_group<M>(J.tab, gi, lane, A0);
    int qn;
    while (true) {
      int nx = min(gi + streams, groups - 1);
      load_group<M>(J.tab, nx, lane, A1);
      m1 = __ldg(J.tab.mask + nx);
      qn = step(A0, gi, m0);
      gi += streams;
      if (gi >= g1 || qn >= 32) break;
      nx = min(gi + streams, groups - 1);
      load_group<M>(J.tab, nx, lane, A0);
      m0 = __ldg(J.tab.mask + nx);
      qn = step(A1, gi, m1);
      gi += streams;
      if (gi >= g1 || qn >= 32) break;
    }
    while (qn >= 32) {
      qn -= 32;
      drain<K>(T, S, J.tab.rows, qn, 32);
    }
    if (gi >= g1 && qn > 0) {
      drain<K>(T, S, J.tab.rows, 0, qn);
      qn = 0;
    }
    if (lane == 0) T.qn[warp] = qn;
    // What the tile's other ranges have found meanwhile.
    if (splits > 1) {
      for (int k = lane; k < 64; k += 32) {
        const int b = hb + k;
        if (!T.live[b]) continue;
        const uint64_t gb = __ldcg(T.gbest + b);
        if (gb < T.seen[b]) {
          T.seen[b] = gb;
          const float th = threshold<K>(T.n2[b], gb, T.sc[b]);
          if (tighter<K>(th, T.ntau[b])) T.ntau[b] = th;
        }
      }
    }
    __syncwarp();
  }
  __syncthreads();
  // The block's best over the warps (and, when split, over the seed ranges).
  uint64_t be = kInfBits;
  uint32_t bs = 0;
  const bool mine = t < nv;
  if (mine) {
    const int wb = wide ? (t >> 6) * 4 : 0;
    for (int k = 0; k < streams; ++k) {
      const uint64_t e = T.best[wb + k][t & 63];
      const uint32_t s = T.bseed[wb + k][t & 63];
      if (s != 0 && (bs == 0 || e < be || (e == be && s < bs))) {
        be = e;
        bs = s;
      }
    }
  }
  if (splits > 1) {
    Part *tp = a.part + (T.sitem0[i] + tile * splits) * kTile + t;  // the tile's records
    if (mine) tp[split * kTile] = Part{be, bs};
    __threadfence();
    __syncthreads();
    if (t == 0) T.last = atomicAdd(a.arrive + stile, 1u) == (uint32_t)(splits - 1);
    __syncthreads();
    if (!T.last) return;
    __threadfence();
    if (mine) {
      be = kInfBits;
      bs = 0;
      for (int k = 0; k < splits; ++k) {
        const uint64_t e = __ldcg(&tp[k * kTile].err);
        const uint32_t s = __ldcg(&tp[k * kTile].seed);
        if (s != 0 && (bs == 0 || e < be || (e == be && s < bs))) {
          be = e;
          bs = s;
        }
      }
    }
  }
  if (mine) write_winner<K>(T, S, J.tab.rows, a.out, t, be, bs);
}

template <bool kLayer>
__global__ void __launch_bounds__(kScreenThreads, 2) k_screen(const __grid_constant__ ScreenArgs a,
                                                              const __grid_constant__ LayerArgs p) {
  extern __shared__ __align__(16) uint8_t smem[];
  TileState &T = *reinterpret_cast<TileState *>(smem);
  if (threadIdx.x == 0) plan_items(T, a, p.R, gridDim.x);
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) T.item = atomicAdd(a.next, 1u);
    __syncthreads();
    const int64_t item = T.item;
    if (item >= T.item0[a.njobs]) return;
    int i = 0;
    while (item >= T.item0[i + 1]) ++i;
    const int64_t local = item - T.item0[i];
    switch (a.job[a.njobs - 1 - i].K) {
      case 2: run_item<2, kLayer>(T, a, p, i, local); break;
      case 3: run_item<3, kLayer>(T, a, p, i, local); break;
      case 4: run_item<4, kLayer>(T, a, p, i, local); break;
      case 5: run_item<5, kLayer>(T, a, p, i, local); break;
      default: run_item<6, kLayer>(T, a, p, i, local); break;
    }
  }
}

// Blocks of each rung before every row: first[j * (R + 1) + r].  One CTA per
// rung, rows in contiguous chunks.
__global__ void __launch_bounds__(1024) k_rung_first(const __grid_constant__ LayerArgs p, int64_t *first) {
  __shared__ int64_t sh[1024];
  const int j = blockIdx.x, t = threadIdx.x, Jm1 = p.J - 1;
  int64_t *out = first + (int64_t)j * (p.R + 1);
  const int64_t per = (p.R + 1023) / 1024, r0 = min((int64_t)t * per, p.R), r1 = min(r0 + per, p.R);
  auto count = [&](int64_t r) {
    const int lo = j > 0 ? p.brk[r * Jm1 + j - 1] : 0, hi = j < Jm1 ? p.brk[r * Jm1 + j] : p.nb;
    return (int64_t)(hi - lo);
  };
  int64_t s = 0;
  for (int64_t r = r0; r < r1; ++r) s += count(r);
  sh[t] = s;
  __syncthreads();
  for (int d = 1; d < 1024; d <<= 1) {
    const int64_t v = t >= d ? sh[t - d] : 0;
    __syncthreads();
    sh[t] += v;
    __syncthreads();
  }
  int64_t run = sh[t] - s;
  for (int64_t r = r0; r < r1; ++r) {
    out[r] = run;
    run += count(r);
  }
  if (t == 1023) out[p.R] = sh[1023];
}

// ---------------------------------------------------------------- host side

size_t frag_bytes(int S, int K) { return ((size_t)1 << S) * 16 * (K <= 3 ? K : 8 - K); }
size_t row_bytes(int S, int K) { return ((size_t)1 << S) * 8 * ((K * (K - 1) + 2 * K + 2) / 2 * 2); }

// One device allocation for everything a call needs beside its arguments.
struct Scratch {
  uint8_t *base = nullptr;
  size_t bytes = 0;
  size_t take(size_t n) {
    const size_t o = bytes;
    bytes += (n + 255) / 256 * 256;
    return o;
  }
};

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

template <bool kLayer>
bool screen(ScreenArgs &a, const LayerArgs &p, cudaStream_t st, cudaError_t *e) {
  const int ctas = 2 * sm_count();
  // plan_items makes at most 3 items per CTA and half a tile's worth of
  // rounding more, and at most 256 of a tile.
  const int64_t tiles = (kLayer ? p.R * (int64_t)p.nb : a.nblocks) / kTile + a.njobs;
  a.max_split = tiles * 256 < 6 * (int64_t)ctas ? tiles * 256 : 6 * (int64_t)ctas;
  Scratch sc;
  size_t frag[kMaxJ], rows[kMaxJ], mask[kMaxJ], jump[kMaxJ];
  int table_ctas = 0, max_k = 2;
  for (int j = 0; j < a.njobs; ++j) {
    const int S = a.job[j].S, K = a.job[j].K;
    frag[j] = sc.take(frag_bytes(S, K));
    rows[j] = sc.take(row_bytes(S, K));
    mask[j] = sc.take(4 * ((size_t)1 << S >> 4));
    jump[j] = sc.take(8 * 512);
    a.job[j].taps = seedq_lfsr_taps(S);
    a.job[j].cta0 = table_ctas;
    table_ctas += (1 << S) / kTableThreads;
    max_k = K > max_k ? K : max_k;
  }
  const size_t first_all = sc.take(kLayer ? 8 * (size_t)a.njobs * (p.R + 1) : 0);
  const size_t part = sc.take(sizeof(Part) * kTile * a.max_split);
  const size_t gbest_bytes = 8 * (size_t)kTile * (tiles < a.max_split ? tiles : a.max_split);
  const size_t gbest = sc.take(gbest_bytes);
  const size_t zeroed = 4 * (size_t)(a.max_split + 2);  // arrive, next, nwide
  const size_t arrive = sc.take(zeroed);
  const size_t wide = sc.take(4 * (size_t)table_ctas * kTableThreads);
  *e = cudaMallocAsync((void **)&sc.base, sc.bytes, st);
  if (*e != cudaSuccess) (void)cudaGetLastError();
  if (*e == cudaErrorMemoryAllocation) return false;
  if (*e != cudaSuccess) return true;  // not a lack of memory: the caller reports it
  for (int j = 0; j < a.njobs; ++j) {
    a.job[j].tab = SeedTables{reinterpret_cast<uint2 *>(sc.base + frag[j]),
                              reinterpret_cast<uint32_t *>(sc.base + mask[j]),
                              reinterpret_cast<double *>(sc.base + rows[j]),
                              reinterpret_cast<uint64_t *>(sc.base + jump[j])};
    a.job[j].first =
        kLayer ? reinterpret_cast<const int64_t *>(sc.base + first_all) + (int64_t)j * (p.R + 1) : nullptr;
  }
  a.part = reinterpret_cast<Part *>(sc.base + part);
  a.gbest = reinterpret_cast<uint64_t *>(sc.base + gbest);
  a.arrive = reinterpret_cast<uint32_t *>(sc.base + arrive);
  a.next = a.arrive + a.max_split;
  a.nwide = a.next + 1;
  a.wide = reinterpret_cast<uint32_t *>(sc.base + wide);
  *e = cudaMemsetAsync(sc.base + arrive, 0, zeroed, st);
  if (*e == cudaSuccess) *e = cudaMemsetAsync(sc.base + gbest, 0x7f, gbest_bytes, st);
  if (*e == cudaSuccess) {
    if (kLayer) k_rung_first<<<a.njobs, 1024, 0, st>>>(p, reinterpret_cast<int64_t *>(sc.base + first_all));
    switch (max_k) {
      case 2: k_seed_tables<2><<<table_ctas, kTableThreads, 0, st>>>(a, p.R); break;
      case 3: k_seed_tables<3><<<table_ctas, kTableThreads, 0, st>>>(a, p.R); break;
      case 4: k_seed_tables<4><<<table_ctas, kTableThreads, 0, st>>>(a, p.R); break;
      case 5: k_seed_tables<5><<<table_ctas, kTableThreads, 0, st>>>(a, p.R); break;
      default: k_seed_tables<6><<<table_ctas, kTableThreads, 0, st>>>(a, p.R); break;
    }
    k_seed_tables_wide<<<sm_count(), kTableThreads, 0, st>>>(a);
    *e = cudaGetLastError();
  }
  // Per call: the attribute belongs to the current device.
  if (*e == cudaSuccess)
    *e = cudaFuncSetAttribute(k_screen<kLayer>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TileState));
  if (*e == cudaSuccess) {
    k_screen<kLayer><<<ctas, kScreenThreads, sizeof(TileState), st>>>(a, p);
    *e = cudaGetLastError();
  }
  const cudaError_t f = cudaFreeAsync(sc.base, st);
  if (*e == cudaSuccess) *e = f;
  return true;
}

}  // namespace

bool screen_blocks(int S, int K, const float *w, int64_t nblocks, const EncodeOut &o, cudaStream_t st,
                   cudaError_t *e) {
  ScreenArgs a = {};
  a.njobs = 1;
  a.job[0].S = S;
  a.job[0].K = K;
  a.out = o;
  a.w = w;
  a.nblocks = nblocks;
  const LayerArgs none = {};
  return screen<false>(a, none, st, e);
}

bool screen_layer(const seedq_layer *L, const float *W, const EncodeOut &o, cudaStream_t st, cudaError_t *e) {
  ScreenArgs a = {};
  a.njobs = L->args.J;
  for (int j = 0; j < a.njobs; ++j) {
    a.job[j].S = L->S[j];
    a.job[j].K = L->k[j];
  }
  a.out = o;
  a.W = W;
  return screen<true>(a, L->args, st, e);
}

}  // namespace seedq
