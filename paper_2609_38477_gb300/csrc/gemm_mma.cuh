// The batch products (n >= 5) of the fused kernel on the tensor cores.
// Included by gemv.cu.
//
// Products of four block columns as m16n8k8 TF32 steps with fp32 accumulation,
// K one weight pair of each.  Lane (g, q) of a warp decodes blocks of column
// c + q and holds their weights where the fragments want them, so nothing is
// transposed or stored: of a block's eight weights the pair (2p, 2p + 1) goes
// into step p.  Up to eight batch entries: M sixteen rows (g and g + 8 of the
// lane's), N the batch, four steps a block.  Up to sixteen: M the batch, N
// eight rows, eight steps a block but half the live weights (the other way
// round 303 us instead of 272 at b16).  A warp takes 32 rows and loads the
// activations of its four columns once for them.
//
// Precision: a weight is an integer of at most 21 bits times a power of two.
// It is split into its top 11 significant bits and the rest (at most 10 bits):
// both are exact in TF32, as is a bfloat16 activation, so every product is
// exact.  A step's eight products are summed by the tensor core, which
// truncates its fp32 result; the four steps of the top parts start from zero
// (the first from the low parts' sum) and are added to fp32 registers by
// ordinary rounding adds, those once per stage to the row's sums, and these
// over the column parts and CTAs with their rounding errors carried along.
// Measured error against fp64, relative to the output's norm, here and in the
// FMA kernel: 0.44e-7 / 0.61e-7 at 64 columns, 0.67e-7 / 0.91e-7 at 1024,
// 0.75e-7 / 1.1e-7 at 4096, 0.84e-7 / 1.3e-7 at 11008 (in one chain of eight
// steps and plain sums 1.3e-7 at 1024).
//
// Work split: a superblock is four row groups (128 rows, in the plan's row
// order); the units (tensor, superblock, column) form one sequence, cut into
// one range of equal modeled cost per CTA.  A CTA takes a superblock's part of
// its range in windows of three stages: its twelve warps are four groups times
// three stages, and the window's activations (bfloat16, permuted by the
// pre-kernel) are copied once for all four groups.  Partial sums of the three
// column parts are added in part order; superblocks cut between CTAs leave
// partial sums in scratch, and the CTA that arrives last adds them in CTA
// order (up to 80 of them, four outputs a thread and eight loads in flight).
//
// Bound by issue (46% to 52% of cycles, 125 instructions per 32 blocks at k = 2,
// 150 at k = 3; ALU 40% to 45%, tensor pipe 14% to 19%): the reconstruction, the split
// (8 logic and 8 packed fp32 instructions a block) and rows that change rung at
// different columns.  The FMA kernel issued 253 at b16, 96 of them products and
// activation loads.  Measured on one GB300 against it: a 7B layer at 4.0 bits,
// b16 381 -> 260 us; two 70B layers at 3.0 bits, b8 1935 -> 1530 us.  Tried:
// masked and unmasked segments of a pass apart (3% to 5% slower), eight warps
// with 242 registers (3% faster at b16, 8% slower at b8), sixteen warps with
// 128 (14% slower), the 11-bit and 10-bit parts in separate sums (equal).
#pragma once

namespace seedq {

constexpr int kMmWarps = 12;
constexpr int kMmThreads = 32 * kMmWarps;
constexpr int kMmParts = kMmWarps / kMmGroups;    // column parts
constexpr int kMmRows = 32 * kMmGroups;

template <int NB>
struct MmCfg {
  static_assert(NB == 8 || NB == 16, "smaller batches run on the FMA pipes");
  static constexpr int ST = 24;                   // columns per stage
  static constexpr int ACC = NB == 16 ? 16 : 8;   // sums a lane holds
  static constexpr int XW = ST * kMmParts;        // columns per window
  static constexpr int PIECES = (ST * 44 / 8 + 12 + 30 + 15) / 16 + 1;
  static constexpr int RW = (PIECES % 2) ? PIECES * 4 : PIECES * 4 + 4;
  static constexpr int STREAM_BYTES = 2 * 32 * RW * 4;   // per warp, double-buffered
  // Bytes of a column's activations: NB x 8 bfloat16, padded so that the
  // fragment loads of four neighbouring columns fall into different banks.
  static constexpr int XCOL = NB * 16 + 32;
  static constexpr int XBYTES = XW * XCOL;               // per window
  static constexpr int COMB_BYTES = kMmParts * kMmRows * NB * 4;
  static constexpr int SMEM = kTableSlots * 4096 + kMmWarps * STREAM_BYTES +
                              (2 * XBYTES > COMB_BYTES ? 2 * XBYTES : COMB_BYTES);
};

__device__ __forceinline__ void mma_tf32(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_tf32_zero(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                              uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// A block's weights, split: pair p's top 11 significant bits and the rest.
struct MmSplit {
  uint64_t top[4], low[4];
};
template <int K>
__device__ __forceinline__ void mm_split(const uint32_t *w, uint32_t pos, bool act, const uint64_t *tab,
                                         const RungDn<K> &rc, MmSplit &o) {
  const uint32_t lo = __funnelshift_r(w[0], w[1], pos), hi = __funnelshift_r(w[1], w[2], pos);
  uint64_t I2[4];
  float scale;
  reconstruct_dn<K>(lo, hi, tab, rc, I2, scale);
  scale = act ? scale : 0.f;
  const uint64_t s2 = f2_pack(scale, scale * (1.0f / (float)(1 << RungDn<K>::Ko)));
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const uint64_t v = f2_mul(I2[p], s2);  // powers of two: exact
    o.top[p] = v & 0xffffe000ffffe000ull;
    o.low[p] = f2_fma(o.top[p], 0xbf800000bf800000ull, v);  // v - top: exact
  }
}

// One rung's pass over columns [clo, chi) of the warp's 32 rows.  Row 8s + g
// has this rung in [ra[s], rb[s]); elsewhere its weights count as zero.  kUni:
// all rows have it in [clo, chi); then only columns past chi have to count as
// zero, which their activations do (the bits read for them are the row's
// next).  Block c of the row starts at bit pb[s] + L c of its staged bytes (row
// r at rows + r * RW words).  xs: the window's activations, column 0 at xs.
template <int K, int NB, bool kUni>
__device__ __forceinline__ void mm_cols(const uint4 *rent, const uint32_t *rows, const int (&pb)[4],
                                        const int (&ra)[4], const int (&rb)[4], int clo, int chi,
                                        const uint64_t *tab, const uint8_t *xs, float (&acc)[MmCfg<NB>::ACC]) {
  using CF = MmCfg<NB>;
  const RungDn<K> rc(rent);
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const int L = (int)rc.S + 4 * K + 4;
  for (int c = clo; c < chi; c += 4) {
    const int col = c + q;
    // Activations of batch g (and g + 8) at the lane's column, bfloat16
    // widened: a weight pair's two per step.
    uint32_t xv[NB == 16 ? 2 : 1][8];
    {
      const uint8_t *xp = xs + min(col, chi - 1) * CF::XCOL + g * 16;
      const bool in = !kUni || col < chi;
#pragma unroll
      for (int t = 0; t < (NB == 16 ? 2 : 1); ++t) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (in) v = *reinterpret_cast<const uint4 *>(xp + 128 * t);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          xv[t][2 * p] = w[p] << 16;
          xv[t][2 * p + 1] = w[p] & 0xffff0000u;
        }
      }
    }
    auto active = [&](int s) { return kUni || (uint32_t)(col - ra[s]) < (uint32_t)(rb[s] - ra[s]); };
    auto split = [&](int s, bool act, MmSplit &o) {
      const uint32_t pos = act ? (uint32_t)(pb[s] + L * col) : 0u;
      mm_split<K>(rows + (8 * s + g) * CF::RW + (pos >> 5), pos, act, tab, rc, o);
    };
    if constexpr (NB == 16) {
      // M the batch, N eight rows: the weights are the B fragment.
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const bool act = active(s);
        // (Eight rows reach a rung later or leave it earlier than the others.)
        if (!kUni && !__any_sync(0xffffffffu, act)) continue;
        MmSplit o;
        split(s, act, o);
        float d[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const uint32_t b0 = (uint32_t)o.low[p], b1 = (uint32_t)(o.low[p] >> 32);
          if (p == 0) mma_tf32_zero(d, xv[0][0], xv[1][0], xv[0][1], xv[1][1], b0, b1);
          else mma_tf32(d, xv[0][2 * p], xv[1][2 * p], xv[0][2 * p + 1], xv[1][2 * p + 1], b0, b1);
        }
        float t[3][4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const uint32_t b0 = (uint32_t)o.top[p], b1 = (uint32_t)(o.top[p] >> 32);
          if (p == 0) mma_tf32(d, xv[0][0], xv[1][0], xv[0][1], xv[1][1], b0, b1);
          else mma_tf32_zero(t[p - 1], xv[0][2 * p], xv[1][2 * p], xv[0][2 * p + 1], xv[1][2 * p + 1], b0, b1);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[4 * s + e] += (d[e] + t[0][e]) + (t[1][e] + t[2][e]);
      }
    } else {
      // M sixteen rows, N the batch: the weights are the A fragment.
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const bool act0 = active(2 * h), act1 = active(2 * h + 1);
        if (!kUni && !__any_sync(0xffffffffu, act0 || act1)) continue;
        MmSplit u, v;
        split(2 * h, act0, u);
        split(2 * h + 1, act1, v);
        float d[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          if (p == 0)
            mma_tf32_zero(d, (uint32_t)u.low[0], (uint32_t)v.low[0], (uint32_t)(u.low[0] >> 32),
                          (uint32_t)(v.low[0] >> 32), xv[0][0], xv[0][1]);
          else
            mma_tf32(d, (uint32_t)u.low[p], (uint32_t)v.low[p], (uint32_t)(u.low[p] >> 32),
                     (uint32_t)(v.low[p] >> 32), xv[0][2 * p], xv[0][2 * p + 1]);
        }
        float t[3][4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const uint32_t a0 = (uint32_t)u.top[p], a1 = (uint32_t)v.top[p], a2 = (uint32_t)(u.top[p] >> 32),
                         a3 = (uint32_t)(v.top[p] >> 32);
          if (p == 0) mma_tf32(d, a0, a1, a2, a3, xv[0][0], xv[0][1]);
          else mma_tf32_zero(t[p - 1], a0, a1, a2, a3, xv[0][2 * p], xv[0][2 * p + 1]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[4 * h + e] += (d[e] + t[0][e]) + (t[1][e] + t[2][e]);
      }
    }
  }
}

// Sign of weight `at` of row r (0, 1 or -1), from its block's fields.
__device__ __forceinline__ int mm_sign(const TensorArgs &T, const int32_t *bk, uint64_t roff, int at) {
  const LayerArgs &p = T.p;
  const int c = at >> 3, i = at & 7, g = rung_of(bk, p.J, c);
  const int S = rung_S(p.code[g]), K = rung_K(p.code[g]);
  const uint64_t off = roff + bits_before(bk, p.J, p.L, p.nb, c);
  if ((off >> 5) + 3 > T.stream_bytes / 4) {
    atomicOr(p.flags, 1u);
    return 0;
  }
  uint32_t lo, hi;
  load_bits<3>(p.stream, off, lo, hi);
  const uint64_t f = ((uint64_t)hi << 32) | lo;
  const uint64_t *tab = p.tables + p.slot[g] * 512;
  const uint32_t seed = lo & ((1u << S) - 1u);
  const uint64_t Q = tab[seed & 255u] ^ tab[256 + (seed >> 8)];
  int I = 0;
  for (int j = 0; j < K; ++j) {
    const int m = (int)(((uint32_t)(f >> (S + 4 + 4 * j)) & 15u) ^ 8u) - 8;
    I += m * ((int)((uint32_t)(Q >> (i * K + j)) & ((1u << S) - 1u)) - (1 << (S - 1)));
  }
  return (I > 0) - (I < 0);
}

// Outputs of batch entries whose activations are not all finite, for the rows
// of superblock sb.  The tensor cores return a NaN for every row of such an
// entry (a zero weight of an inactive rung times an infinity), so its outputs
// follow from the row's own products instead: a NaN activation makes each of
// them NaN, an infinite one adds an infinity of the weight's sign, or a NaN
// where the weight is zero.  A warp per entry looks through its activations and
// lists the infinite ones, kList at a time; a thread then reads the signs of
// its row's weights there, until two differ.  An entry that is all finite
// overflowed, and keeps its sums.
// bad: bit b for an output of entry b that the thread found not finite; list:
// kList NB words.
// Measured, a 7B layer with one NaN or infinity in one entry, against a row
// walked by one thread per output: b8 26,300 -> 289 us, b16 49,700 -> 336 us
// (all finite 251 and 280); every activation NaN at b16 62,000 -> 351 us.
template <int NB>
__device__ __noinline__ void mm_nonfinite(const TensorArgs &T, const uint16_t *X, float *Y, int64_t sb, uint32_t bad,
                                          uint32_t *list) {
  constexpr int kList = kMmParts * kMmRows;  // of each entry: all together fill the parts' sums
  constexpr int kEach = (NB + kMmParts - 1) / kMmParts;  // entries per thread
  static_assert(kMmThreads == kMmParts * kMmRows, "thread (part, row)");
  __shared__ uint32_t s_bad, s_nan, s_inf;   // bits: entries looked at, with a NaN, with an infinity
  __shared__ int s_count[NB], s_next[NB];    // listed, block the next round starts at (nb: no more)
  const LayerArgs &p = T.p;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nb = p.nb;
  if (t == 0) s_bad = s_nan = s_inf = 0u;
  if (t < NB) s_next[t] = 0;
  __syncthreads();
  if (bad) atomicOr(&s_bad, bad);
  const int64_t pos = sb * kMmRows + t % kMmRows;
  const bool mine = pos < p.R;
  const int64_t r = mine ? __ldg(p.rowperm + pos) : 0;
  int32_t bk[kMaxJ];
  for (int j = 0; j < p.J - 1; ++j) bk[j] = __ldg(p.brk + r * (p.J - 1) + j);
  const uint64_t roff = __ldg(p.row_off + r);
  __syncthreads();
  const uint32_t entries = s_bad;
  uint32_t plus = 0u, minus = 0u;  // bit k: an infinity of that sign in the row's entry t / kMmRows + kMmParts k
  bool more = true;
  for (bool first = true; more; first = false) {
    for (int b = warp; b < NB; b += kMmWarps) {
      if (!(entries >> b & 1u)) continue;
      const uint4 *xv = reinterpret_cast<const uint4 *>(p.xperm) + b;
      int count = 0, next = nb;
      bool nan = false, inf = false;
#pragma unroll 4
      for (int c0 = s_next[b]; c0 < nb; c0 += 32) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (c0 + lane < nb) v = __ldg(xv + (int64_t)(c0 + lane) * NB);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        uint32_t hit = 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint32_t h = (w[i >> 1] >> (16 * (i & 1))) & 0x7fffu;
          nan = nan || h > 0x7f80u;
          hit |= (uint32_t)(h == 0x7f80u) << i;
        }
        if (!__any_sync(0xffffffffu, hit != 0u)) continue;
        inf = true;
        if (next == nb && count + 256 > kList) next = c0;
        if (next < nb && !first) break;  // (the first round looks for a NaN in all of them)
        if (next < nb) continue;
        int at = __popc(hit);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v2 = __shfl_up_sync(0xffffffffu, at, o);
          if (lane >= o) at += v2;
        }
        const int total = __shfl_sync(0xffffffffu, at, 31);
        at += count - __popc(hit);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (hit >> i & 1u)
            list[b * kList + at++] = (uint32_t)((c0 + lane) * 8 + i) | ((w[i >> 1] >> (16 * (i & 1) + 15) & 1u) << 31);
        count += total;
      }
      nan = __any_sync(0xffffffffu, nan);
      if (lane == 0) {
        s_count[b] = first && nan ? 0 : count;
        s_next[b] = first && nan ? nb : next;
        if (first && nan) atomicOr(&s_nan, 1u << b);
        if (first && inf) atomicOr(&s_inf, 1u << b);
      }
    }
    __syncthreads();
    more = false;
    for (int k = 0; mine && k < kEach; ++k) {
      const int b = t / kMmRows + kMmParts * k;
      if (b >= NB || !(entries >> b & 1u)) continue;
      const int count = s_count[b];
      for (int i = 0; i < count && !((plus & minus) >> k & 1u); ++i) {
        const uint32_t e = list[b * kList + i];
        const int sg = mm_sign(T, bk, roff, (int)(e & 0x7fffffffu));
        if (sg >= 0) (e >> 31 ? minus : plus) |= 1u << k;
        if (sg <= 0) (e >> 31 ? plus : minus) |= 1u << k;
      }
      more = more || (s_next[b] < nb && !((plus & minus) >> k & 1u));
    }
    more = __syncthreads_or(more) != 0;
  }
  for (int k = 0; mine && k < kEach; ++k) {
    const int b = t / kMmRows + kMmParts * k;
    if (b >= NB || !((s_nan | s_inf) >> b & 1u)) continue;
    const float inf = __int_as_float(0x7f800000);
    const bool nan = (s_nan | (((plus & minus) >> k & 1u) << b)) >> b & 1u;
    Y[(int64_t)b * p.R + r] = (nan ? inf - inf : minus >> k & 1u ? -inf : inf) + outlier_term(p, X, r, b);
  }
  __syncthreads();
}

// Sum of partial sums with the rounding errors of its additions (Knuth's
// two-sum).  An overflow stays the infinity it is.
struct MmSum {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float t = __fadd_rn(s, v), z = __fsub_rn(t, s);
    e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(v, z)));
    s = t;
  }
  __device__ __forceinline__ float value() const { return isfinite(s) ? __fadd_rn(s, e) : s; }
};

// T, and where it is a kernel parameter its copy in the CTA's shared memory, for
// code out of line: taken by address there it costs the main loop its constant
// operands (a 7B layer at b8 235 -> 239 us).
template <bool kSet>
__device__ __forceinline__ const TensorArgs &mm_shared(const TensorArgs &T, TensorArgs &sT) {
  if constexpr (kSet) return T;
  __syncthreads();
  if (threadIdx.x == 0) sT = T;
  __syncthreads();
  return sT;
}

// Output i (row, batch entry) of a superblock from the column parts' sums.
template <int NB>
__device__ __forceinline__ float mm_parts(const float *comb, int i) {
  MmSum sum;
#pragma unroll
  for (int k = 0; k < kMmParts; ++k) sum.add(comb[k * kMmRows * NB + i]);
  return sum.value();
}

// y of a superblock that one CTA has whole.
template <int NB, bool kSet>
__device__ __forceinline__ void mm_write(const TensorArgs &T, int n, const uint16_t *X, float *Y, int64_t sb, float *comb,
                                         TensorArgs &sT) {
  const LayerArgs &p = T.p;
  const int64_t row0 = sb * kMmRows;
  // The rows' places are loaded ahead of the sums, all at once (four 8B layers
  // at 3.0 bits and b16 919 -> 907 us).
  constexpr int kEach = (kMmRows * NB + kMmThreads - 1) / kMmThreads;
  int32_t rr[kEach];
#pragma unroll
  for (int k = 0; k < kEach; ++k) {
    const int row = (threadIdx.x + k * kMmThreads) / NB;
    rr[k] = row < kMmRows && row0 + row < p.R ? __ldg(p.rowperm + row0 + row) : -1;
  }
  uint32_t bad = 0u;
#pragma unroll
  for (int k = 0; k < kEach; ++k) {
    const int i = threadIdx.x + k * kMmThreads, b = i % NB;
    if (rr[k] < 0 || b >= n) continue;
    const float v = mm_parts<NB>(comb, i);
    if (!isfinite(v)) bad |= 1u << b;
    Y[(int64_t)b * p.R + rr[k]] = v + outlier_term(p, X, rr[k], b);
  }
  if (__syncthreads_or(bad != 0u)) mm_nonfinite<NB>(mm_shared<kSet>(T, sT), X, Y, sb, bad, reinterpret_cast<uint32_t *>(comb));
}

// The CTA's partial sums of a cut superblock (tensor T, superblock sb) are in
// its slots: counts the CTA's arrival, and where it is the last, adds all of
// them in CTA order and writes y.  No CTA waits for another.
template <int NB, bool kSet>
__device__ __forceinline__ void mm_finish(const TensorArgs &T, const int64_t *cb, int ctas, int n, const uint16_t *X,
                                          float *Y, int64_t sb, uint32_t *list, TensorArgs &sT) {
  __shared__ int s_last;
  const LayerArgs &p = T.p;
  const int64_t gu = T.ubegin_mm + sb * p.nb;
  const int cf = cta_of(cb, ctas, gu), cl = cta_of(cb, ctas, gu + p.nb - 1);
  __syncthreads();  // (the last call's s_last)
  if (threadIdx.x == 0) s_last = atomicAdd(p.counters + sb, 1) == cl - cf;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // The first CTA's range may start before this superblock, the others' start in
  // it.  Four neighbouring outputs per thread, kAhead CTAs' sums in flight.
  constexpr int kAhead = 8, kPiece = kMmRows * NB / 4;
  const float4 *slots = reinterpret_cast<const float4 *>(p.slots);
  const float4 *first = slots + ((int64_t)cf * 2 + (cb[cf] >= gu ? 0 : 1)) * kPiece;
  const float4 *rest = slots + (int64_t)(cf + 1) * 2 * kPiece;
  const int others = cl - cf;
  uint32_t bad = 0u;
  for (int i = threadIdx.x; i < kPiece; i += kMmThreads) {
    const int row = i / (NB / 4), b0 = i % (NB / 4) * 4;
    const int64_t pos = sb * kMmRows + row;
    if (pos >= p.R) continue;
    MmSum sum[4];
    auto add = [&](const float4 &v) {
      sum[0].add(v.x);
      sum[1].add(v.y);
      sum[2].add(v.z);
      sum[3].add(v.w);
    };
    add(__ldcg(first + i));
    const float4 *at = rest + i;
    int c = 0;
    for (; c + kAhead <= others; c += kAhead, at += 2 * kAhead * kPiece) {
      float4 v[kAhead];
#pragma unroll
      for (int k = 0; k < kAhead; ++k) v[k] = __ldcg(at + 2 * k * kPiece);
#pragma unroll
      for (int k = 0; k < kAhead; ++k) add(v[k]);
    }
    for (; c < others; ++c, at += 2 * kPiece) add(__ldcg(at));
    const int64_t rr = __ldg(p.rowperm + pos);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int b = b0 + e;
      if (b >= n) continue;
      const float v = sum[e].value();
      if (!isfinite(v)) bad |= 1u << b;
      Y[(int64_t)b * p.R + rr] = v + outlier_term(p, X, rr, b);
    }
  }
  if (__syncthreads_or(bad != 0u)) mm_nonfinite<NB>(mm_shared<kSet>(T, sT), X, Y, sb, bad, list);
  if (threadIdx.x == 0) p.counters[sb] = 0;
}

template <int NB, bool kSet>
__global__ void __launch_bounds__(kMmThreads, 1) k_gemm(const __grid_constant__ MultiArgs a) {
  using CF = MmCfg<NB>;
  extern __shared__ __align__(16) uint64_t smem[];
  uint64_t *tabs = smem;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gi = warp % kMmGroups, part = warp / kMmGroups;
  uint8_t *base = reinterpret_cast<uint8_t *>(smem + kTableSlots * 512);
  uint32_t *sbuf = reinterpret_cast<uint32_t *>(base + warp * CF::STREAM_BYTES);
  uint8_t *xbuf = base + kMmWarps * CF::STREAM_BYTES;
  float *comb = reinterpret_cast<float *>(xbuf);  // after a piece's last window
  __shared__ TensorArgs sT;
  __shared__ uint4 rdn[kMaxJ * RungDn<2>::kEntry];
  __shared__ int cut_ti[2];
  __shared__ int64_t cut_sb[2];
  {
    // The jump tables depend only on S, so any tensor's copy serves all.
    const uint4 *src = reinterpret_cast<const uint4 *>((kSet ? a.tens : a.t)[0].p.tables);
    uint4 *dst = reinterpret_cast<uint4 *>(tabs);
    for (int i = threadIdx.x; i < kTableSlots * 256; i += kMmThreads) dst[i] = __ldg(src + i);
  }
  // The permuted activations come from the pre-kernel launched just before.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int cta = blockIdx.x;
  const TensorArgs *tens = kSet ? a.tens : a.t;
  const int64_t *cb = kSet ? a.cbd : a.cta_begin;
  const int64_t u0 = cb[cta], u1 = cb[cta + 1];
  int ti = 0;
  {
    int lo = 0, hi = a.nt - 1;  // last tensor whose first unit is <= u0
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (tens[mid].ubegin_mm <= u0) lo = mid;
      else hi = mid - 1;
    }
    ti = lo;
  }
  // Superblocks cut where the range starts and ends (tensor -1: none).
  if (threadIdx.x < 2) cut_ti[threadIdx.x] = -1;
  for (int64_t u = u0; u < u1;) {
    while (ti + 1 < a.nt && tens[ti + 1].ubegin_mm <= u) ++ti;
    __syncthreads();  // the last piece is done with sT, rdn and the buffers
    if constexpr (kSet) {
      const uint32_t *srcw = reinterpret_cast<const uint32_t *>(tens + ti);
      uint32_t *dstw = reinterpret_cast<uint32_t *>(&sT);
      for (int w = threadIdx.x; w < (int)(sizeof(TensorArgs) / 4); w += kMmThreads) dstw[w] = srcw[w];
    }
    store_rung_entries(tens[ti].p, a.zero, rdn);
    __syncthreads();
    const TensorArgs &T = kSet ? sT : a.t[ti];
    const LayerArgs &p = T.p;
    const int nb = p.nb, J = p.J;
    const int64_t lu = u - T.ubegin_mm, tend = (ti + 1 < a.nt) ? tens[ti + 1].ubegin_mm : cb[a.ctas];
    const int64_t sb = lu / nb;
    const int ca = (int)(lu - sb * nb), ce_piece = (int)min((int64_t)nb, ca + (min(u1, tend) - u));
    const int cbk = ce_piece;
    // The lane's row of the warp's group (rows past R repeat the group's
    // first; groups past the last repeat nothing and do no work).
    const int64_t r0 = (sb * kMmGroups + gi) * 32;
    const bool have = r0 < p.R;
    const int64_t ridx = have ? (r0 + lane < p.R ? r0 + lane : r0) : 0;
    const uint4 m0 = __ldg(p.rowrec + 2 * ridx), m1 = __ldg(p.rowrec + 2 * ridx + 1);
    const uint64_t roff = (uint64_t)m0.x | ((uint64_t)m0.y << 32);
    const uint32_t bw[4] = {m0.z, m0.w, m1.x, m1.y};
    const uint8_t *gstream = reinterpret_cast<const uint8_t *>(p.stream);
    const int windows = (cbk - ca + CF::XW - 1) / CF::XW;
    // A part's columns of the window at w0: whole stages, the piece's last
    // window in even shares (multiples of the four columns of a step).
    auto part_cols = [&](int w0, int &cs, int &ce) {
      const int share = min(CF::ST, ((cbk - w0 + kMmParts - 1) / kMmParts + 3) & ~3);
      cs = w0 + part * share;
      ce = min(cbk, cs + share);
    };
    int p0_of[2] = {0, 0};  // staged bit position of block 0 of the row's rung 0 (may be negative)
    auto issue = [&](int v) {
      const int b = v & 1;
      // Activations of the window, one 16-byte piece (a column's batch entry)
      // at a time.
      const int w0 = ca + v * CF::XW, wn = min(cbk, w0 + CF::XW) - w0;
      const uint8_t *xsrc = reinterpret_cast<const uint8_t *>(p.xperm) + (int64_t)w0 * NB * 16;
      uint8_t *xdst = xbuf + b * CF::XBYTES;
      for (int i = threadIdx.x; i < wn * NB; i += kMmThreads)
        cp_async16(reinterpret_cast<float *>(xdst + (i / NB) * CF::XCOL + (i % NB) * 16),
                   xsrc + (int64_t)i * 16);
      int cs, ce;
      part_cols(w0, cs, ce);
      if (have && cs < ce) {
        uint32_t s_cs, s_ce;
        lane_bits_before(bw, p, cs, ce, s_cs, s_ce);
        // A row's last stage ends where its record says the row ends.
        if (ce == nb && s_ce != m1.z) atomicOr(p.flags, 1u);
        const uint64_t bit_cs = roff + s_cs;
        const uint64_t b_lo = (bit_cs >> 3) & ~(uint64_t)15;
        uint64_t b_hi = (roff + s_ce + 96 + 7) >> 3;
        b_hi = (b_hi + 15) & ~(uint64_t)15;
        if (b_hi > T.stream_bytes) {
          // The plan disagrees with the bound buffer: read what is there, report it.
          atomicOr(p.flags, 1u);
          b_hi = T.stream_bytes & ~(uint64_t)15;
        }
        const int npc = b_hi > b_lo ? (int)min((uint64_t)CF::PIECES, (b_hi - b_lo) >> 4) : 0;
        const int p0 = (int)((int64_t)roff - (int64_t)(b_lo * 8));
        if (b) p0_of[1] = p0;
        else p0_of[0] = p0;
        uint32_t *rows = sbuf + b * 32 * CF::RW + lane * CF::RW;
#pragma unroll
        for (int pc = 0; pc < CF::PIECES; ++pc)
          if (pc < npc) cp_async16(rows + pc * 4, gstream + b_lo + 16 * pc);
      }
      cp_async_commit();
    };
    float tot[CF::ACC];
#pragma unroll
    for (int i = 0; i < CF::ACC; ++i) tot[i] = 0.f;
    // The first rung some row still has at the warp's stage (they rise), each
    // row's first column at it, and the bits its blocks there start later than
    // at rung 0's rate.
    int j0 = 0, from0 = 0, off0 = 0;
    auto brk_of = [&](int j) {
      if (j >= J - 1) return nb;
      uint32_t wv = bw[0];
      wv = (j >> 1) == 1 ? bw[1] : (j >> 1) == 2 ? bw[2] : (j >> 1) == 3 ? bw[3] : wv;
      return (int)((wv >> (16 * (j & 1))) & 0xffffu);
    };
    issue(0);
    for (int v = 0; v < windows; ++v) {
      // This thread's copies of window v are done; after the barrier every
      // thread's are, and no warp is still in window v - 1, whose buffers the
      // next copies fill.
      cp_async_wait<0>();
      __syncthreads();
      if (v + 1 < windows) issue(v + 1);
      const int b = v & 1;
      const int w0 = ca + v * CF::XW;
      int cs, ce;
      part_cols(w0, cs, ce);
      if (!have || cs >= ce) continue;
      const uint8_t *xs = xbuf + b * CF::XBYTES - (int64_t)w0 * CF::XCOL;
      const uint32_t *rows = sbuf + b * 32 * CF::RW;
      float acc[CF::ACC];
#pragma unroll
      for (int i = 0; i < CF::ACC; ++i) acc[i] = 0.f;
      while (j0 < J - 1) {
        const int to = brk_of(j0);
        if (!__all_sync(0xffffffffu, to <= cs)) break;
        off0 -= p.dL[j0] * to;
        from0 = to;
        ++j0;
      }
      // Rung by rung: the row's columns at rung j, the bits before them.
      int from = from0, posb = (b ? p0_of[1] : p0_of[0]) + off0;
      for (int j = j0; j < J; ++j) {
        const int to = brk_of(j);
        const int lo = max(cs, from), hi = min(ce, to);
        const unsigned any = __ballot_sync(0xffffffffu, lo < hi);
        if (any) {
          const int clo = __reduce_min_sync(0xffffffffu, lo < hi ? lo : 0x7fffffff);
          const int chi = __reduce_max_sync(0xffffffffu, lo < hi ? hi : 0);
          int pb[4], ra[4], rb[4];
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            const int src = 8 * s + (lane >> 2);
            pb[s] = __shfl_sync(0xffffffffu, posb, src);
            ra[s] = __shfl_sync(0xffffffffu, lo, src);
            rb[s] = max(__shfl_sync(0xffffffffu, hi, src), ra[s]);
          }
          const uint4 *rent = rdn + j * RungDn<2>::kEntry;
          const uint64_t *tab = tabs + p.slot[j] * 512;
          const bool uni = __all_sync(0xffffffffu, lo == clo && hi == chi);
          switch (rung_K(p.code[j]) * 2 + uni) {
#define MM_CASE(K)                                                                              \
  case 2 * K: mm_cols<K, NB, false>(rent, rows, pb, ra, rb, clo, chi, tab, xs, acc); break;     \
  case 2 * K + 1: mm_cols<K, NB, true>(rent, rows, pb, ra, rb, clo, chi, tab, xs, acc); break;
            MM_CASE(2)
            MM_CASE(3)
            MM_CASE(4)
            MM_CASE(5)
            MM_CASE(6)
#undef MM_CASE
          }
        } else if (__all_sync(0xffffffffu, from >= ce)) {
          break;
        }
        // Block c of rung j + 1 starts dL[j] (c - to) bits later than at rung j's rate.
        if (j < J - 1) posb -= p.dL[j] * to;
        from = to;
      }
#pragma unroll
      for (int i = 0; i < CF::ACC; ++i) tot[i] += acc[i];
    }
    __syncthreads();  // the window buffers become the parts' sums
    // Sums of a part: comb[part][row][batch].
    {
      const int g = lane >> 2, q = lane & 3;
      float *cg = comb + (part * kMmGroups + gi) * 32 * NB;
      if constexpr (NB == 16) {  // lane (g, q): batch g and g + 8 of rows 8s + 2q and 8s + 2q + 1
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          float *cr = cg + (8 * s + 2 * q) * NB + g;
          cr[0] = tot[4 * s];
          cr[NB] = tot[4 * s + 1];
          cr[8] = tot[4 * s + 2];
          cr[NB + 8] = tot[4 * s + 3];
        }
      } else {  // batch 2q and 2q + 1 of rows 16h + g and 16h + g + 8
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float *cr = cg + (16 * h + g) * NB + 2 * q;
          *reinterpret_cast<float2 *>(cr) = make_float2(tot[4 * h], tot[4 * h + 1]);
          *reinterpret_cast<float2 *>(cr + 8 * NB) = make_float2(tot[4 * h + 2], tot[4 * h + 3]);
        }
      }
    }
    __syncthreads();
    const bool full = ca == 0 && cbk == nb;
    const int side = u == u0 ? 0 : 1;
    if (full) {
      mm_write<NB, kSet>(T, a.n, kSet ? a.Xall + (int64_t)a.n * T.cpre : T.x, kSet ? a.Yall + (int64_t)a.n * T.rpre : T.y,
                   sb, comb, sT);
    } else {
      float *slot = p.slots + ((int64_t)cta * 2 + side) * kMmRows * NB;
      for (int i = threadIdx.x; i < kMmRows * NB; i += kMmThreads) slot[i] = mm_parts<NB>(comb, i);
      if (threadIdx.x == 0) {
        cut_ti[side] = ti;
        cut_sb[side] = sb;
      }
    }
    u += cbk - ca;
  }
  __threadfence();
  __syncthreads();
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    const int ci = cut_ti[side];
    if (ci < 0) continue;
    const TensorArgs &T = tens[ci];
    mm_finish<NB, kSet>(T, cb, a.ctas, a.n, kSet ? a.Xall + (int64_t)a.n * T.cpre : T.x,
                  kSet ? a.Yall + (int64_t)a.n * T.rpre : T.y, cut_sb[side],
                  reinterpret_cast<uint32_t *>(comb), sT);
  }
}

// Activations for the tensor-core path: bfloat16 in permuted column order,
// zero at outlier columns and past n, xperm[(c * NB + b) * 8 + i] =
// x_b[perm[8 c + i]].  One thread per (block column, batch entry).
__device__ __forceinline__ void xperm_bf16(const int32_t *perm, const uint16_t *x, uint4 *out, int64_t C, int n_out,
                                           const int32_t *out_cols, int n, int nbt) {
  const int64_t total = C / 8 * nbt;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = t / nbt;
    const int b = (int)(t - c * nbt);
    uint32_t v[4] = {0u, 0u, 0u, 0u};
    if (b < n) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int col = __ldg(perm + 8 * c + i);
        bool outl = false;
        for (int o = 0; o < n_out; ++o) outl |= out_cols[o] == col;
        const uint32_t h = outl ? 0u : (uint32_t)__ldg(x + (int64_t)b * C + col);
        v[i >> 1] |= h << (16 * (i & 1));
      }
    }
    out[t] = make_uint4(v[0], v[1], v[2], v[3]);
  }
}

}  // namespace seedq
