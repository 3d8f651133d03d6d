// Alg. 2 in full: materialize W_hat (rows of it) in the original column order.
//
// Two kernels.  k_decode_tile builds whole rows in shared memory, where the
// scatter through the inverse permutation costs bank conflicts, and writes
// them out as one contiguous bulk copy.  k_decode scatters straight to memory,
// four bytes to a 32-byte sector: it takes the outputs that are small, or of
// short rows, where that is the faster (tile_is_faster), rows too long for
// shared memory and outputs that are not 16-byte aligned.
#include <cuda_fp16.h>

#include <algorithm>

#include "device_once.h"
#include "seedq_internal.cuh"

namespace seedq {

template <int K>
__device__ __forceinline__ void decode_block(const LayerArgs &p, int S, uint64_t off,
                                             const uint64_t *tab, float *Wrow, int c) {
  uint32_t lo, hi;
  load_bits<3>(p.stream, off, lo, hi);  // the stream buffer ends in 16 bytes of slack
  float I[8], scale;
  const RungRt<K> rc(S, p.zero);
  reconstruct_rt<K>(lo, hi, tab, rc, I, scale);
#pragma unroll
  for (int i = 0; i < 8; ++i) Wrow[__ldg(p.perm + 8 * c + i)] = I[i] * scale;  // exact
}

// One thread per block, straight to memory; reads l(g_b) bits at the block's offset (row offset +
// closed form over the row's rung breakpoints), writes 8 weights through the
// inverse permutation (the scatter step of Alg. 2).
__global__ void __launch_bounds__(256) k_decode(const __grid_constant__ LayerArgs p, int64_t row0, int64_t nrows, float *W) {
  const int64_t total = nrows * (int64_t)p.nb;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < total;
       b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = b / p.nb;
    const int c = (int)(b - i * p.nb);
    const int64_t r = row0 + i;
    int32_t bk[kMaxJ];
    for (int j = 0; j < p.J - 1; ++j) bk[j] = __ldg(p.brk + r * (p.J - 1) + j);
    const int g = rung_of(bk, p.J, c);
    const uint64_t roff = __ldg(p.row_off + r);
    const uint64_t off = roff + bits_before(bk, p.J, p.L, p.nb, c);
    // The plan and the bound buffer must agree: the last block of a row ends
    // at the next row's offset, and the block's three words are readable.
    // Otherwise flag bit 0 and leave the block's weights unwritten.
    if (c == p.nb - 1 && off + (uint64_t)p.L[g] != __ldg(p.row_off + r + 1)) atomicOr(p.flags, 1u);
    if ((off >> 5) + 3 > p.stream_words) {
      atomicOr(p.flags, 1u);
      continue;
    }
    const uint64_t *tab = p.tables + (size_t)p.slot[g] * 512;
    float *Wrow = W + i * p.C;
    const int S = rung_S(p.code[g]);
    switch (rung_K(p.code[g])) {
      case 2: decode_block<2>(p, S, off, tab, Wrow, c); break;
      case 3: decode_block<3>(p, S, off, tab, Wrow, c); break;
      case 4: decode_block<4>(p, S, off, tab, Wrow, c); break;
      case 5: decode_block<5>(p, S, off, tab, Wrow, c); break;
      case 6: decode_block<6>(p, S, off, tab, Wrow, c); break;
      default: atomicOr(p.flags, 1u);
    }
  }
}

// Outlier columns overwrite the codec's values (Alg. 2 last step; Sec. 3.5).
__global__ void k_outliers(const __grid_constant__ LayerArgs p, int64_t row0, int64_t nrows, float *W) {
  const int64_t total = nrows * p.n_out;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = t / p.n_out;
    const int o = (int)(t - i * p.n_out);
    const uint16_t h = p.out_vals[(row0 + i) * p.n_out + o];
    W[i * p.C + p.out_cols[o]] = __half2float(__ushort_as_half(h));
  }
}

// ------------------------------------------------------------ whole rows
//
// One CTA per SM takes tiles of consecutive rows (contiguous in W and in the
// stream).  Its last warp copies the tiles' stream bytes in a few tiles ahead
// (cp.async.bulk on an mbarrier, with the rows' records) and, when the decoding
// warps have all arrived on a second mbarrier, writes the finished tile out
// with one bulk copy and hands the buffer back on a third.  The decoding warps
// so wait neither for memory nor for the slowest of them.  A warp decodes 32
// neighbouring blocks of a row at a time and scatters their weights through
// the permutation (16-bit copy in shared memory).  Outlier columns are
// overwritten in the buffer by the thread that wrote them.
//
// Bound by issue (63% of cycles) and the shared-memory pipe (61%: the scatter's
// eight random words a block, two table lookups, the rung's constants), ahead
// of the 4 bytes a weight written.  Measured against k_decode on one GB300:
// 4096 x 11008 with a row factor and four outlier columns 287 -> 71 us (2.8
// TB/s of weights and stream), 4096 x 4096 94 -> 32, 1024 x 1040 9.2 -> 7.6,
// 512 x 20000 64 -> 29.
// On the way: two 512-thread CTAs per SM with barriers around each tile 88 us;
// the moving warp instead of barriers 80; stream and permutation in shared
// memory 80; chunks dealt from where the last tile ended 72 (the warps with
// the odd chunk of every row had been the slow ones).  960 decoding threads
// (64 registers, spills) 76, 608 72.5.
constexpr int kDecThreads = 736;                // decoding threads (80 registers); one more warp moves data
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kDecRows = 32;                    // rows per tile at most
constexpr int kDecStages = 4;                   // tiles whose stream bytes are in flight or in use
constexpr int kDecSmemMax = 227 * 1024;

struct __align__(16) DecRow {
  int32_t bk[kMaxJ - 1];    // breakpoints, kMaxCols past J - 1
  int32_t base[kMaxJ];      // block c of rung g starts at staged bit base[g] + L[g] c
  int32_t end;              // staged bit of the next row
  uint32_t words;           // staged words of the tile
  uint64_t word0;           // the tile's first staged word in the stream
};

struct DecFixed {
  uint64_t tabs[kTableSlots * 512];
  uint4 rdn[kMaxJ * RungDn<2>::kEntry];
  uint4 rung[kMaxJ];                 // L, K, first table entry
  DecRow row[kDecStages][kDecRows];
  uint32_t outl[kMaxCols / 8 / 32];  // nonzero: the 32 blocks hold an outlier column
  uint64_t ready[kDecStages];        // mbarriers: a stage's stream bytes and records are in place
  uint64_t full[2];                  // per buffer: every decoding warp is through with the tile
  uint64_t free_[2];                 // per buffer: its tile has been read for the copy out
};

__device__ __forceinline__ void mbar_init(uint64_t *b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"((uint32_t)__cvta_generic_to_shared(b)) : "memory");
}
// Waits for the phase of the given parity; false after about a second.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity) {
  for (int i = 0; i < (1 << 20); ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2, 1000;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(done) : "r"((uint32_t)__cvta_generic_to_shared(b)), "r"(parity) : "memory");
    if (done) return true;
  }
  return false;
}

// Rung records of the tile's rows (one lane per row).  Bits relative to the
// staged bytes fit 32 bits: a tile has at most kDecRows * kMaxCols / 8 blocks.
__device__ __forceinline__ void dec_rows(const LayerArgs &p, int64_t r0, int nr, uint64_t word0, uint32_t words,
                                         DecRow *rows) {
  const int l = threadIdx.x & 31;
  if (l >= nr) return;
  // Rung g spans blocks [bk[g-1], bk[g]).
  DecRow &R = rows[l];
  const int64_t r = r0 + l;
  int32_t base = (int32_t)(__ldg(p.row_off + r) - word0 * 32);
  R.base[0] = base;
  R.end = (int32_t)(__ldg(p.row_off + r + 1) - word0 * 32);
  R.word0 = word0;
  R.words = words;
#pragma unroll
  for (int j = 0; j < kMaxJ - 1; ++j) {
    const int bk = j < p.J - 1 ? __ldg(p.brk + r * (p.J - 1) + j) : kMaxCols;
    R.bk[j] = bk;
    base -= p.dL[j] * bk;
    R.base[j + 1] = base;
  }
}

template <int K>
__device__ __forceinline__ void decode_dn(uint32_t lo, uint32_t hi, const uint64_t *tab, const uint4 *rent, float (&w)[8]) {
  const RungDn<K> rc(rent);
  uint64_t I2[4];
  float scale;
  reconstruct_dn<K>(lo, hi, tab, rc, I2, scale);
  // Powers of two: exact.
  const uint64_t s2 = f2_pack(scale, scale * (1.0f / (float)(1 << RungDn<K>::Ko)));
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const float2 v = f2_unpack(f2_mul(I2[p], s2));
    w[2 * p] = v.x;
    w[2 * p + 1] = v.y;
  }
}

// Shared memory behind the fixed part: the permutation, then nbuf buffers of
// trows rows of weights and kDecStages of their stream bytes.
struct DecLayout {
  int trows, nbuf;
  uint32_t buf, buf_bytes, str, str_bytes, total;
};
constexpr uint32_t kDecFixed = (sizeof(DecFixed) + 127) / 128 * 128;

__host__ __device__ inline uint32_t dec_stream_bytes(int trows, int nb) {
  // Blocks of at most 44 bits, the last one's read-ahead and the alignment.
  return (uint32_t)(((int64_t)trows * nb * 44 / 8 + 12 + 32 + 127) / 128 * 128);
}

static DecLayout dec_layout(int64_t C, int trows, int nbuf) {
  DecLayout l;
  l.trows = trows;
  l.nbuf = nbuf;
  l.buf_bytes = (uint32_t)((trows * C * 4 + 127) / 128 * 128);
  l.str_bytes = dec_stream_bytes(trows, (int)(C / 8));
  l.buf = (uint32_t)((kDecFixed + 2 * C + 127) / 128 * 128);
  l.str = l.buf + nbuf * l.buf_bytes;
  l.total = l.str + kDecStages * l.str_bytes;
  return l;
}

__global__ void __launch_bounds__(kDecThreads + 32, 1)
    k_decode_tile(const __grid_constant__ LayerArgs p, int64_t row0, int64_t nrows, float *W, const DecLayout lay) {
  extern __shared__ __align__(128) uint8_t smem[];
  DecFixed &F = *reinterpret_cast<DecFixed *>(smem);
  uint16_t *perm = reinterpret_cast<uint16_t *>(smem + kDecFixed);
  const int t = threadIdx.x, trows = lay.trows, nbuf = lay.nbuf;
  for (int i = t; i < (int)p.C; i += kDecThreads + 32) perm[i] = (uint16_t)__ldg(p.perm + i);
  {
    const uint4 *src = reinterpret_cast<const uint4 *>(p.tables);
    uint4 *dst = reinterpret_cast<uint4 *>(F.tabs);
    for (int i = t; i < kTableSlots * 256; i += kDecThreads + 32) dst[i] = __ldg(src + i);
    for (int i = t; i < kMaxCols / 8 / 32; i += kDecThreads + 32) F.outl[i] = 0u;
    if (t < p.J) F.rung[t] = make_uint4(p.L[t], rung_K(p.code[t]), p.slot[t] * 512, 0u);
  }
  store_rung_entries(p, p.zero, F.rdn);
  if (t == 0) {
    for (int b = 0; b < kDecStages; ++b) mbar_init(F.ready + b, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(F.full + b, kDecWarps);
      mbar_init(F.free_ + b, 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (t < p.n_out) {
    const int c = __ldg(p.invperm + p.out_cols[t]) >> 3;
    F.outl[c >> 5] = 1u;
  }
  __syncthreads();
  const int64_t tiles = (nrows + trows - 1) / trows;
  const int C = (int)p.C;
  if (t >= kDecThreads) {
    // The moving warp.
    auto stage = [&](int64_t tile, int b) {
      if (tile >= tiles) return;
      const int nr = (int)min((int64_t)trows, nrows - tile * trows);
      const int64_t r0 = row0 + tile * trows;
      // The tile's stream bytes: whole 16-byte pieces, cut where the readable
      // buffer ends and at the stage's size.
      const uint64_t lo = (__ldg(p.row_off + r0) >> 3) & ~(uint64_t)15;
      uint64_t hi = (((__ldg(p.row_off + r0 + nr) + 96 + 7) >> 3) + 15) & ~(uint64_t)15;
      hi = min(hi, min(p.stream_words * 4, lo + lay.str_bytes) & ~(uint64_t)15);
      const uint32_t bytes = hi > lo ? (uint32_t)(hi - lo) : 0u;
      dec_rows(p, r0, nr, lo >> 2, bytes >> 2, F.row[b]);
      __syncwarp();
      if (t == kDecThreads) {
        const uint32_t bar = (uint32_t)__cvta_generic_to_shared(F.ready + b);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
        if (bytes)
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                           (uint32_t)__cvta_generic_to_shared(smem + lay.str + b * lay.str_bytes)),
                       "l"(reinterpret_cast<const uint8_t *>(p.stream) + lo), "r"(bytes), "r"(bar)
                       : "memory");
      }
      __syncwarp();
    };
    for (int b = 0; b < kDecStages; ++b) stage(blockIdx.x + (int64_t)b * gridDim.x, b);
    uint32_t b = 0, ph = 0, sb = 0, sph = 0;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      if (!mbar_wait(F.full + b, ph)) {
        // The decoding warps have given up.  Copies into this CTA's shared
        // memory must not outlive it: those of the kDecStages tiles from here.
        atomicOr(p.flags, 1u);
        for (int k = 0; k < kDecStages && tile + (int64_t)k * gridDim.x < tiles; ++k) {
          mbar_wait(F.ready + sb, sph);
          if (++sb == kDecStages) {
            sb = 0;
            sph ^= 1;
          }
        }
        break;
      }
      if (t == kDecThreads) {
        const int64_t n0 = tile * trows;
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(W + n0 * p.C),
                     "r"((uint32_t)__cvta_generic_to_shared(smem + lay.buf + b * lay.buf_bytes)),
                     "r"((uint32_t)(min((int64_t)trows, nrows - n0) * C * 4))
                     : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
      stage(tile + (int64_t)kDecStages * gridDim.x, sb);
      if (t == kDecThreads) {
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        mbar_arrive(F.free_ + b);
      }
      if (++sb == kDecStages) {
        sb = 0;
        sph ^= 1;
      }
      if (++b == (uint32_t)nbuf) {
        b = 0;
        ph ^= 1;
      }
    }
    if (t == kDecThreads) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    return;
  }
  uint32_t b = 0, ph = 0, sb = 0, sph = 0;
  int chunk = t >> 5;  // the warp's first chunk of the tile
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t i0 = tile * trows;
    const int nr = (int)min((int64_t)trows, nrows - i0);
    float *buf = reinterpret_cast<float *>(smem + lay.buf + b * lay.buf_bytes);
    const uint32_t *str = reinterpret_cast<const uint32_t *>(smem + lay.str + sb * lay.str_bytes);
    const DecRow *rows = F.row[sb];
    // (A buffer's first use finds the phase before its first release complete.)
    if (!mbar_wait(F.ready + sb, sph) || !mbar_wait(F.free_ + b, ph ^ 1)) {
      atomicOr(p.flags, 1u);
      return;
    }
    // The tile's rows in chunks of 32 columns, dealt to the warps round-robin
    // from where the last tile's deal ended, so that no warp draws more.
    const int lane = t & 31, cpr = (p.nb + 31) / 32, chunks = nr * cpr;
    for (int k = chunk; k < chunks; k += kDecWarps) {
      const int i = k / cpr, k0 = k - i * cpr, c = k0 * 32 + lane;
      const DecRow &R = rows[i];
      // The chunk's first rung by one compare per lane; a lane past a
      // breakpoint inside the chunk moves on from there.
      int g = __popc(__ballot_sync(0xffffffffu, lane < kMaxJ - 1 && k0 * 32 >= R.bk[lane & 7]));
      while (c >= R.bk[g & 7] && g < kMaxJ - 1) ++g;
      const uint4 rg = F.rung[g];
      const int off = R.base[g] + (int)rg.x * c;
      const uint32_t at = (uint32_t)off >> 5;
      const bool ok = c < p.nb;
      // As k_decode: the plan and the bound buffer must agree.
      if (c == p.nb - 1 && off + (int)rg.x != R.end) atomicOr(p.flags, 1u);
      if (!ok) continue;
      const uint4 pc = *reinterpret_cast<const uint4 *>(perm + 8 * c);
      const uint32_t col[8] = {pc.x & 0xffffu, pc.x >> 16, pc.y & 0xffffu, pc.y >> 16,
                               pc.z & 0xffffu, pc.z >> 16, pc.w & 0xffffu, pc.w >> 16};
      float w[8];
      uint32_t w0, w1, w2;
      bool readable = true;
      if (at + 3 <= R.words) {
        w0 = str[at];
        w1 = str[at + 1];
        w2 = str[at + 2];
      } else {  // the last words of a buffer that is cut short or not a multiple of 16 bytes
        const uint64_t wi = R.word0 + at;
        readable = wi + 3 <= p.stream_words;
        w0 = readable ? __ldg(p.stream + wi) : 0u;
        w1 = readable ? __ldg(p.stream + wi + 1) : 0u;
        w2 = readable ? __ldg(p.stream + wi + 2) : 0u;
      }
      const uint32_t lo = __funnelshift_r(w0, w1, (uint32_t)off), hi = __funnelshift_r(w1, w2, (uint32_t)off);
      const uint64_t *tab = F.tabs + rg.z;
      const uint4 *rent = F.rdn + g * RungDn<2>::kEntry;
      switch (rg.y) {
        case 2: decode_dn<2>(lo, hi, tab, rent, w); break;
        case 3: decode_dn<3>(lo, hi, tab, rent, w); break;
        case 4: decode_dn<4>(lo, hi, tab, rent, w); break;
        case 5: decode_dn<5>(lo, hi, tab, rent, w); break;
        default: decode_dn<6>(lo, hi, tab, rent, w); break;
      }
      float *brow = buf + i * C;
      if (!readable) {
        atomicOr(p.flags, 1u);
        const float *old = W + (i0 + i) * p.C;  // a block that cannot be read keeps what W holds
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = old[col[e]];
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) brow[col[e]] = w[e];
      if (F.outl[k0]) {
        const int first = c * 8;
        for (int o = 0; o < p.n_out; ++o) {
          const int at_o = __ldg(p.invperm + p.out_cols[o]) - first;
          if (at_o >= 0 && at_o < 8)
            brow[p.out_cols[o]] = __half2float(__ushort_as_half(__ldg(p.out_vals + (row0 + i0 + i) * p.n_out + o)));
        }
      }
    }
    chunk -= chunks % kDecWarps;
    if (chunk < 0) chunk += kDecWarps;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if ((t & 31) == 0) mbar_arrive(F.full + b);
    if (++sb == kDecStages) {
      sb = 0;
      sph ^= 1;
    }
    if (++b == (uint32_t)nbuf) {
      b = 0;
      ph ^= 1;
    }
  }
}
static_assert(kDecRows <= 32, "one lane of the storing warp per row record");

// k_decode takes 4.5 us a million weights (the sectors it writes) and, with
// outliers, a second launch.  k_decode_tile takes 0.6 us more to start and then, for
// each row an SM gets, 0.07 us and 0.23 us a thousand columns, its first 40 rows
// 0.13 us more.  Fitted to 500 sizes from 1 x 8 to 60000 x 384 and 8192 x 8192, with
// and without outliers: at most 9% slower than always direct and 12% (0.9 us) than
// always tiles.  Measured, direct / tile: 8 x 22400 4.9 / 10.7 us, 4096 x 64 5.2 /
// 9.1, 8192 x 128 8.4 / 12.3, 4096 x 512 12.9 / 11.1, 1024 x 1040 9.2 / 7.6, 4096 x
// 11008 278 / 68.
static bool tile_is_faster(int64_t rows, int64_t C, int sms, bool outliers) {
  const double weights = (double)rows * (double)C, each = (double)((rows + sms - 1) / sms);
  const double direct = 4.5e-6 * weights + (outliers ? 1.3 + 0.35e-3 * std::min((double)rows, 8000.0) : 0.0);
  const double tile = 0.6 + each * std::max(0.115, 0.07 + 0.23e-3 * (double)C) + 0.13 * std::min(each, 40.0);
  return weights > (outliers ? 1500.0 : 16384.0) && direct > tile;
}

// The kernel's dynamic shared-memory limit is a per-device attribute: set once
// per device, and again if a launch reports an invalid configuration (the
// device's context may have been reset since).
static cudaError_t launch_tile(const LayerArgs &p, int64_t row0, int64_t nrows, float *W, const DecLayout &lay, int dev,
                               int grid, cudaStream_t st) {
  static DeviceOnce once;
  auto limit = [&] {
    return (cudaError_t)once.run(dev, [] {
      return (int)cudaFuncSetAttribute(k_decode_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, kDecSmemMax);
    });
  };
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kDecThreads + 32);
  cfg.dynamicSmemBytes = lay.total;
  cfg.stream = st;
  cudaError_t e = limit();
  if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, k_decode_tile, p, row0, nrows, W, lay);
  if (e == cudaErrorInvalidValue) {
    (void)cudaGetLastError();
    once.forget(dev);
    e = limit();
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, k_decode_tile, p, row0, nrows, W, lay);
  }
  return e;
}

}  // namespace seedq

using namespace seedq;

extern "C" {

seedq_status seedq_decode_rows(const seedq_layer *L, int64_t row0, int64_t nrows, float *W,
                               void *cuda_stream) {
  if (!L || !W || row0 < 0 || nrows < 0 || row0 + nrows > L->args.R) return SEEDQ_ERR_INVALID_ARG;
  if (!L->args.stream) return SEEDQ_ERR_STREAM;
  if (nrows == 0) return SEEDQ_OK;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t C = L->args.C;
  DecLayout lay = dec_layout(C, 1, 2);
  if (lay.total > (uint32_t)kDecSmemMax) lay = dec_layout(C, 1, 1);
  if (((uintptr_t)W & 15u) == 0 && lay.total <= (uint32_t)kDecSmemMax &&
      tile_is_faster(nrows, C, sms, L->args.n_out > 0)) {
    // Rows per tile: as many as fit twice, fewer when each SM would get less
    // than four tiles, but at least a chunk for every decoding warp while that
    // leaves each SM a tile.
    if (lay.nbuf == 2) {
      const int64_t cpr = (L->args.nb + 31) / 32, fill = kDecWarps / cpr, each = (nrows + sms - 1) / sms;
      int64_t rows = nrows / (4 * sms), least = fill < each ? fill : each;
      rows = rows < least ? least : rows;
      rows = rows > kDecRows ? kDecRows : rows;
      while (rows > 1 && dec_layout(C, (int)rows, 2).total > (uint32_t)kDecSmemMax) --rows;
      if (rows > 1) lay = dec_layout(C, (int)rows, 2);
    }
    const int64_t tiles = (nrows + lay.trows - 1) / lay.trows;
    SEEDQ_CUDA(launch_tile(L->args, row0, nrows, W, lay, dev, (int)(tiles < sms ? tiles : sms), st));
    return SEEDQ_OK;
  }
  const int64_t blocks = nrows * (int64_t)L->args.nb;
  const int64_t want = (blocks + 255) / 256;
  const int grid = (int)(want < (int64_t)sms * 16 ? want : (int64_t)sms * 16);
  k_decode<<<grid, 256, 0, st>>>(L->args, row0, nrows, W);
  SEEDQ_CUDA(cudaGetLastError());
  if (L->args.n_out > 0) {
    const int64_t t = nrows * L->args.n_out;
    const int g2 = (int)((t + 255) / 256 < 4096 ? (t + 255) / 256 : 4096);
    k_outliers<<<g2, 256, 0, st>>>(L->args, row0, nrows, W);
    SEEDQ_CUDA(cudaGetLastError());
  }
  return SEEDQ_OK;
}

seedq_status seedq_decode_weights(const seedq_layer *L, float *W, void *cuda_stream) {
  if (!L) return SEEDQ_ERR_INVALID_ARG;
  return seedq_decode_rows(L, 0, L->args.R, W, cuda_stream);
}

}  // extern "C"
