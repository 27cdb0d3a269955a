// xengine.cu -- the X-engine CMAC kernel for sm_103a (tcgen05 + TMA + TMEM).
//
// For one channel, the X-engine (Sec. 2.3) forms V[i][j] = sum_t x_i conj(x_j)
// over the lower triangle (Eq. 1, Eq. 2).  With x = a + j b:
//   Re V_ij = sum_t a_i a_j + b_i b_j   = <[a_i, b_i], [a_j, b_j]>
//   Im V_ij = sum_t b_i a_j - a_i b_j   = <[b_i, -a_i], [a_j, b_j]>
// so with K running over (t, re/im) the whole channel is one real matrix
// product D = Arows * Brows^T, where every input contributes an "A row"
// [a, b] (used on both sides) and a "Q row" [b, -a] (row side only).  That is
// a dense rank-2T update, so it runs on the tensor cores: 8-bit float operands
// and fp32 accumulators in TMEM.  The operands are E4M3 bytes of the biased
// values u = v + 8, 0 <= u <= 15 (E4M3 is linear there: byte u is u 2^-9), so
// a nibble becomes an operand byte by one logic operation; 15 operations for
// four samples' A and Q rows became 4 (192 inputs, 1024 channels, 8 blocks of
// 8192 samples with the dump: 5.85 -> 4.88 ms).  The epilogue takes the bias
// out exactly with the rows' sums of u, which the unpack warps accumulate:
//   sum (u_i - 8)(u_j - 8) = sum u_i u_j - 8 sum u_i - 8 sum u_j + 64 T.
// A sample adds at most 2 x 225 units of 2^-18 to an accumulator and an item
// spans at most 32768 samples, so every fp32 partial is an integer below 2^24
// (times 2^-18) and exact; each item's sums are folded into the int64
// integration buffer when it ends.
//
// What bounds it at 192 inputs: the MMAs on shared-memory operands.  One of N
// columns takes about 24 + N / 2 cycles per 32-byte K slice (57 at N = 64, 155
// at 256), so the three strips take about 1056 of a 64-sample chunk's 1100 to
// 1130 cycles (256 channels, 8 blocks of 8192 samples: 943 to 978 us a launch
// at 1.99 GHz; without the decode 8 % less).  Other sizes: see chunk_cost in
// xe_sched.h.
//
// Kernel structure (persistent, one CTA per SM, 28 warps):
//   warp 24     TMA producer: packed bytes [channel][input][time] -> smem ring
//   warps 0-15  unpack: 4-bit nibbles -> E4M3 A/Q rows in the 128B-swizzled
//               K-major layout the MMA reads (the paper's CPU "fluff" step,
//               Sec. 2.3, moved on chip)
//   warps 25-27 MMA issuers: tcgen05.mma M=128 (64 inputs' A rows + Q rows),
//               N = columns of the triangle strip, K = 32 per instruction;
//               one issuing thread per accumulator, because a single thread
//               issues an MMA only every ~110-126 cycles in a loop with
//               waits and commits, too slow for the N = 64 strips alone
//   warps 16-23 epilogue: tcgen05.ld of the fp32 accumulators, bias out,
//               rows regrouped through a small buffer, int64 red.add into the
//               lower triangle (256 contiguous bytes an instruction)
// A launch integrates up to kMaxBlocksPerLaunch blocks; the host cuts its
// items at fold windows of at most 32768 samples.
// A work unit is (problem, template, channel); a template names the inputs
// staged per chunk and the MMAs (row tile x column range) that cover its part
// of the triangle.  The host cuts the units into items (a unit over a range
// of 128-sample stages) and deals them to the CTAs in shares of about equal
// cost, so the last wave does not leave SMs idle; a launch may
// hold several independent problems (a batch of correlators).  All waits are
// bounded by a timeout; on expiry the kernel drains its own copies and MMAs,
// frees TMEM and reports through *status.
// The Gram instance (GRAM, up to 128 inputs) keeps an input's real and
// imaginary parts in rows of their own, 128 samples to a row, and accumulates
// the four kinds of product apart: half the operand bytes, no negated rows, one
// hand-off per 128 samples, twice the accumulator columns.  (128 inputs, 512
// channels, 4 blocks of 8192 samples: 741 -> 567 us a launch; 64 inputs, 8
// blocks: 824 -> 612; 16 inputs: 237 -> 179.)
// At 72 registers a thread every instance spills a little (bytes stored /
// loaded: one CTA 12 / 12, pair 20 / 28, Gram 44 / 116, F-engine order 48 / 56,
// Gram in F-engine order 68 / 144, pair in F-engine order 84 / 140).
// The CTA-pair instance (PAIR) runs clusters of two CTAs on two SMs: each
// stages and unpacks two row tiles and half of a B operand of up to 256
// columns, the even CTA's two issuers run M = 256 MMAs (cta_group::2) over
// both halves and commit to both CTAs' barriers, one thread of the odd CTA
// forwards its unpack warps' stage arrivals to the even CTA, and each CTA
// folds its own 128 TMEM lanes.
#include <cuda.h>

#include <cstring>

#include "ptx.cuh"
#include "xe_internal.h"
#include "xe_sched.h"
#include "xe_unpack.cuh"

namespace xe {

namespace {

struct Bars {
  uint32_t pk_full, pk_empty, z_full, z_empty, acc_full, acc_empty, drain, never;
  // the table of operand sums: complete (unpack warps), cleared (epilogue),
  // and read by every epilogue warp
  uint32_t sum_full, sum_empty, sum_read;
};

}  // namespace

// Item `it` of the launch (explicit list, or derived from the unit index).
__device__ __forceinline__ XItem item_at(const XParams &p, int it) {
  if (p.items) return p.items[it];
  XItem r;
  r.prob = 0;
  const int unit = it / p.implicit_nseg, seg = it - unit * p.implicit_nseg;
  r.tpl = unit / p.implicit_n_chan;
  r.chan = (unit - r.tpl * p.implicit_n_chan) * p.implicit_chan_step;
  r.pk0 = (int)((long long)p.implicit_npk * seg / p.implicit_nseg);
  r.npk = (int)((long long)p.implicit_npk * (seg + 1) / p.implicit_nseg) - r.pk0;
  return r;
}

// Walks the packed stages of an item through its blocks: stage kc of the
// block (a division once per item instead of one per stage and role).
struct StageWalk {
  int kc, pk_per_block, last;  // last: chunks in a block's last stage
  __device__ __forceinline__ StageWalk(const XProb &pb, int pk0)
      : kc(pk0 % pb.pk_per_block),
        pk_per_block(pb.pk_per_block),
        last(pb.chunks_per_block - kChunksPerPk * (pb.pk_per_block - 1)) {}
  // chunks (of kChunkSamples) in this stage
  __device__ __forceinline__ int chunks() const {
    return kc == pk_per_block - 1 ? last : kChunksPerPk;
  }
  // to the next stage; true if it is the first of the next block
  __device__ __forceinline__ bool next() {
    if (++kc < pk_per_block) return false;
    kc = 0;
    return true;
  }
};

// Decodes this warp's rows of one chunk of a staged region: n_k groups of 8
// rows, 64 rows apart.  `src` and `dst` are the lane's addresses in the first
// group; Q: Q rows are stored 1024 bytes (eight operand rows) after the A
// rows.  The sums of u go to the halves of sum[k].
template <bool Q>
__device__ __forceinline__ void unpack_rows(uint32_t src, uint32_t dst, uint32_t dst_step, int n_k,
                                            uint32_t (&sum)[4]) {
  constexpr uint32_t kStep = kTileInputs * kPackedRowBytes;
  uint4 in[2];
  in[0] = lds128(src);
  if (n_k > 1) in[1] = lds128(src + kStep);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (k >= n_k) break;
    const uint4 x = in[k & 1];
    if (k + 2 < n_k) in[k & 1] = lds128(src + (uint32_t)(k + 2) * kStep);
    const uint32_t d0 = dst + (Q ? (uint32_t)k * 16384u : (uint32_t)k * dst_step), d1 = d0 ^ 16u;
    uint32_t re0, im0, nre0, re1, im1, nre1, re2, im2, nre2, re3, im3, nre3;
    decode_biased(x.x, re0, im0, nre0);
    decode_biased(x.y, re1, im1, nre1);
    decode_biased(x.z, re2, im2, nre2);
    decode_biased(x.w, re3, im3, nre3);
    sts128(d0, re0, im0, re1, im1);
    sts128(d1, re2, im2, re3, im3);
    if (Q) {
      sts128_q(d0, im0, nre0, im1, nre1);
      sts128_q(d1, im2, nre2, im3, nre3);
    }
    sum[k] = __dp4a(re0 + re1 + re2 + re3, 0x01010101u, sum[k]) +
             (__dp4a(im0 + im1 + im2 + im3, 0x01010101u, 0u) << 16);
  }
}

// The same for a region in F-engine order: each 64-input box is [128
// samples][64 inputs].  Item (qd, j) of a box: inputs 4 qd .. 4 qd + 3,
// samples 8 j .. 8 j + 7 of the chunk; eight 4-byte loads (one sample of four
// inputs each), two 4 x 4 byte transposes, and per input two decoded words:
// 16 bytes of its A row (and Q row) at K bytes 16 j .. 16 j + 15.  The
// half-warp of odd j loads its samples rotated by one (the same rotation for
// every input, so a fixed permutation of K), which puts the two half-warps'
// rows on different bank halves.  Within every 8-input group of a region the
// operand row of group position pos is (pos + group) % 8: the eight threads
// of a store phase then hit eight bank groups.  Thread t of the group takes
// item t % 128 of boxes t / 128 and t / 128 + 2.
__device__ __forceinline__ void unpack_turned(uint32_t src, uint32_t dst, int kind, int n_box,
                                              int t, int sub, uint32_t (&sum)[8]) {
  const int v = t & 127, qd = v & 15, j = v >> 4, jj = j & 1;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int box = 2 * k + (t >> 7);
    if (box >= n_box) break;
    const uint32_t at =
        src + (uint32_t)box * 8192u + (uint32_t)(64 * (kChunkSamples * sub + 8 * j)) + 4u * qd;
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = lds32(at + 64u * (uint32_t)((i + jj) & 7));
    uint32_t lo[4], hi[4];
    transpose4(w[0], w[1], w[2], w[3], lo[0], lo[1], lo[2], lo[3]);
    transpose4(w[4], w[5], w[6], w[7], hi[0], hi[1], hi[2], hi[3]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      uint32_t re_l, im_l, nre_l, re_h, im_h, nre_h;
      decode_biased(lo[e], re_l, im_l, nre_l);
      decode_biased(hi[e], re_h, im_h, nre_h);
      sum[4 * k + e] = __dp4a(re_l + re_h, 0x01010101u, sum[4 * k + e]) +
                       (__dp4a(im_l + im_h, 0x01010101u, 0u) << 16);
      const int i_rel = kTileInputs * box + 4 * qd + e, gp = i_rel >> 3;
      const int pos = ((i_rel & 7) + (gp & 3)) & 7;
      const uint32_t d = dst + (uint32_t)((kind ? 16 : 8) * gp + pos) * 128u +
                         (uint32_t)((j ^ pos) << 4);
      sts128(d, re_l, im_l, re_h, im_h);
      if (kind == 1) sts128_q(d, im_l, nre_l, im_h, nre_h);
    }
  }
}
// The Gram form of unpack_rows: 128 samples of this warp's rows, the lane's two
// 16-sample chunks (g and g + 4) one after the other.  The real bytes go to the
// same 16-byte chunk of the first operand row, the imaginary ones to the second
// (1024 bytes on): half of the stores of unpack_rows<true>.
__device__ __forceinline__ void unpack_gram(uint32_t src, uint32_t dst, int n_k,
                                            uint32_t (&sum)[4]) {
#pragma unroll
  for (int k = 0; k < 2; ++k) {  // at most two tiles of a region
    if (k >= n_k) break;
    const uint32_t s0 = src + (uint32_t)(k * kTileInputs * kPackedRowBytes);
    const uint32_t d0 = dst + (uint32_t)k * 16384u;
    const uint4 x[2] = {lds128(s0), lds128(s0 ^ 64u)};
    uint32_t re = 0u, im = 0u;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      uint32_t re0, im0, re1, im1, re2, im2, re3, im3, n;
      decode_biased(x[c].x, re0, im0, n);
      decode_biased(x[c].y, re1, im1, n);
      decode_biased(x[c].z, re2, im2, n);
      decode_biased(x[c].w, re3, im3, n);
      sts128(d0 ^ (64u * c), re0, re1, re2, re3);
      sts128_q(d0 ^ (64u * c), im0, im1, im2, im3);
      re += re0 + re1 + re2 + re3;  // bytes: at most 8 x 15
      im += im0 + im1 + im2 + im3;
    }
    sum[k] = __dp4a(re, 0x01010101u, sum[k]) + (__dp4a(im, 0x01010101u, 0u) << 16);
  }
}

// The Gram form of unpack_turned: item (qd, j) is inputs 4 qd .. 4 qd + 3 and
// samples 16 j .. 16 j + 15 of the stage, with the same rotations.
__device__ __forceinline__ void unpack_gram_turned(uint32_t src, uint32_t dst, int n_box, int t,
                                                   uint32_t (&sum)[8]) {
  const int v = t & 127, qd = v & 15, j = v >> 4, jj = j & 1;
  const int box = t >> 7;  // at most two boxes of a region
  if (box >= n_box) return;
  const uint32_t at = src + (uint32_t)box * 8192u + (uint32_t)(64 * 16 * j) + 4u * qd;
  uint32_t w[4][4];  // [input][4 samples]
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    uint32_t x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = lds32(at + 64u * (uint32_t)((4 * m + i + jj) & 15));
    transpose4(x[0], x[1], x[2], x[3], w[0][m], w[1][m], w[2][m], w[3][m]);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    uint32_t re[4], im[4], n;
#pragma unroll
    for (int m = 0; m < 4; ++m) decode_biased(w[e][m], re[m], im[m], n);
    const int i_rel = kTileInputs * box + 4 * qd + e, gp = i_rel >> 3;
    const int pos = ((i_rel & 7) + (gp & 3)) & 7;
    const uint32_t d = dst + (uint32_t)(16 * gp + pos) * 128u + (uint32_t)((j ^ pos) << 4);
    sts128(d, re[0], re[1], re[2], re[3]);
    sts128_q(d, im[0], im[1], im[2], im[3]);
    sum[e] = __dp4a(re[0] + re[1] + re[2] + re[3], 0x01010101u, sum[e]) +
             (__dp4a(im[0] + im[1] + im[2] + im[3], 0x01010101u, 0u) << 16);
  }
}

// A folded value from an accumulator (in units of 2^-18) and the sum of its
// operand-sum entries, given plus kMagicBits: acc 2^18 - 8 sum, returned plus
// kMagicBits.  1.5 x 2^23 has a unit of 1, so adding a whole number below 2^22
// to its bits or to its value is the same thing; the entries stay below 2^20,
// folded values within 128 x 32768 = 2^22, and all steps are exact.  (Four
// quick operations; the conversion instruction takes eight cycles a warp.)
constexpr uint32_t kMagicBits = 0x4B400000u;  // 1.5 x 2^23
__device__ __forceinline__ uint32_t unbias(uint32_t acc, uint32_t sum_magic) {
  constexpr float kMagic = 12582912.0f;
  const float bias = fmaf(__uint_as_float(sum_magic), -8.0f, 8.0f * kMagic);
  return __float_as_uint(fmaf(__uint_as_float(acc), 262144.0f, bias) + kMagic);
}

// kThreads = 32 * 28: warps 0-15 unpack, 16-23 epilogue, 24 TMA, 25-27 MMA.
// Every role walks the same item list, [cta_first[b], cta_first[b + 1]).
// TCN: the blocks are in F-engine order (XParams::tcn), staged and unpacked
// by the transposing path; a compile-time choice, so that the X-engine-order
// kernel carries none of that code.
// PAIR: the launch is clusters of two CTAs running pair units (XUnit::
// pair_rows): both CTAs stage and unpack their own rows, the even CTA's
// issuers run M = 256 MMAs over both, and both fold their own TMEM rows.
// GRAM: units of the Gram form (XUnit::gram).
template <int M, bool TCN, bool PAIR, bool GRAM>
__global__ void __launch_bounds__(kThreads, 1)
    xengine_cmac_kernel(const __grid_constant__ XMapsT<M> maps, const XParams p) {
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte alignment for the swizzled operand atoms
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t *z_buf = smem;
  uint8_t *pk_buf = z_buf + (size_t)p.z_stages * p.z_stage_bytes;
  uint64_t *bar_mem = reinterpret_cast<uint64_t *>(pk_buf + (size_t)p.pk_stages * p.pk_stage_bytes);
  // [pk_full x S][pk_empty x S][z_full x Z][z_empty x Z][acc_full][acc_empty][drain x kMmaWarps]
  // [never]: only waited on by the failure-detection self-test
  // [sum_full][sum_empty][sum_read]
  uint32_t *misc = reinterpret_cast<uint32_t *>(bar_mem + 2 * p.pk_stages + 2 * p.z_stages + 2 +
                                                kMmaWarps + 1 + 3);
  // behind the barrier area: the epilogue warps' buffers, then the table of
  // operand sums (p.sum_rows entries of 8 bytes)
  uint8_t *epi_mem = reinterpret_cast<uint8_t *>(bar_mem) + kBarrierBytes;
  uint8_t *sum_mem = epi_mem + kEpiWarps * kEpiBufBytes;
  volatile int *abort_flag = reinterpret_cast<volatile int *>(misc + 1);
  const uint32_t bar0 = smem_u32(bar_mem);
  Bars b;
  b.pk_full = bar0;
  b.pk_empty = bar0 + 8 * p.pk_stages;
  b.z_full = bar0 + 16 * p.pk_stages;
  b.z_empty = b.z_full + 8 * p.z_stages;
  b.acc_full = b.z_empty + 8 * p.z_stages;
  b.acc_empty = b.acc_full + 8;
  b.drain = b.acc_empty + 8;
  b.never = b.drain + 8 * kMmaWarps;
  b.sum_full = b.never + 8;
  b.sum_empty = b.sum_full + 8;
  b.sum_read = b.sum_empty + 8;
  const uint32_t tab = smem_u32(sum_mem);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.pk_stages; ++s) {
      mbar_init(b.pk_full + 8 * s, 1);
      mbar_init(b.pk_empty + 8 * s, kUnpackWarps);
    }
    for (int s = 0; s < p.z_stages; ++s) {
      // a pair's even CTA also counts the odd CTA's forwarded arrive
      mbar_init(b.z_full + 8 * s, (PAIR && cluster_ctarank() == 0) ? kUnpackGroup + 1 : kUnpackGroup);
      mbar_init(b.z_empty + 8 * s, PAIR ? kPairIssuers : kMmaWarps);
    }
    mbar_init(b.acc_full, PAIR ? kPairIssuers : kMmaWarps);
    mbar_init(b.acc_empty, PAIR ? 2 * kEpiWarps : kEpiWarps);
    for (int m = 0; m < kMmaWarps; ++m) mbar_init(b.drain + 8 * m, 1);
    mbar_init(b.never, 1);  // nothing ever arrives here
    mbar_init(b.sum_full, (PAIR ? 2 : 1) * kUnpackWarps);
    mbar_init(b.sum_empty, (PAIR ? 2 : 1) * kEpiWarps);
    mbar_init(b.sum_read, kEpiWarps);
    *abort_flag = 0;
    fence_mbar_init();
  }
  // the unpack warps add to the table of operand sums, starting from zero
  for (int k = threadIdx.x; k < 2 * p.sum_rows; k += kThreads)
    reinterpret_cast<uint32_t *>(sum_mem)[k] = 0u;
  if (warp == kWarpMma0) {
    if (PAIR) {
      tmem_alloc_pair(smem_u32(misc), kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(misc), kTmemCols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  // a pair's CTAs arrive on each other's barriers: both must be initialised
  if (PAIR) cluster_sync();
  tc_fence_after();
  const uint32_t tmem = misc[0];
  // rank in the pair (the odd CTA stages its regions from in_lo1 and owns
  // its segments' rows from row_in1)
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;

  int it0, it1, it_step;
  if (p.items) {
    const int wkr = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;  // cluster or CTA
    it0 = p.cta_first[wkr];
    it1 = p.cta_first[wkr + 1];
    it_step = 1;
  } else {
    it0 = blockIdx.x;
    it1 = p.implicit_n_tpl * p.implicit_n_chan * p.implicit_nseg;
    it_step = gridDim.x;
  }
  const uint64_t to = p.timeout_ns;

  if (warp == kWarpTma) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      int armed[kMaxPkStages];
      uint32_t armed_ph[kMaxPkStages];
      for (int k = 0; k < kMaxPkStages; ++k) armed[k] = 0, armed_ph[k] = 0;
      bool ok = true;
      int last_map = -1;
      for (int it = it0; it < it1 && ok && !*abort_flag; it += it_step) {
        const XItem item = item_at(p, it);
        const XProb pb = p.probs[item.prob];
        const XUnit *u = pb.units + item.tpl;
        const int n_reg = u->n_reg;
        const uint32_t bytes = (uint32_t)u->pk_bytes;
        StageWalk walk(pb, item.pk0);
        int mi = pb.map0 + item.pk0 / pb.pk_per_block;
        for (int k = 0; k < item.npk; ++k) {
          const int kc = walk.kc;
          const void *tmap = &maps.m[mi][0];
          if (mi != last_map) { prefetch_tmap(tmap); last_map = mi; }
          if (!mbar_wait(b.pk_empty + 8 * s, ph ^ 1u, abort_flag, to)) { ok = false; break; }
          const uint32_t full = b.pk_full + 8 * s;
          mbar_arrive_expect_tx(full, bytes);
          armed[s] = 1;
          armed_ph[s] = ph;
          const uint32_t dst0 = smem_u32(pk_buf + (size_t)s * p.pk_stage_bytes);
          for (int r = 0; r < n_reg; ++r) {
            const int in_lo = rank ? u->reg[r].in_lo1 : u->reg[r].in_lo, n_in = u->reg[r].n_in;
            const int off = u->reg[r].pk_off;
            // past the last channel: zero fill (also where the sum wraps around)
            const int ch = (int)((uint32_t)item.chan + (uint32_t)u->reg[r].chan_off);
            for (int bx = 0; bx < n_in; bx += kTileInputs) {
              if (TCN)  // (input, channel, time): a [128 samples][64 inputs] box
                tma_load_3d(dst0 + off + bx * kPackedRowBytes, tmap, full, in_lo + bx, ch,
                            kc * kPkSamples);
              else        // (time, input, channel): a [64 inputs][128 samples] box
                tma_load_3d(dst0 + off + bx * kPackedRowBytes, tmap, full, kc * kPkSamples,
                            in_lo + bx, ch);
            }
          }
          if (walk.next()) ++mi;
          if (++s == p.pk_stages) { s = 0; ph ^= 1u; }
        }
      }
      // every load this thread armed must have landed before the CTA exits
      int dummy = 0;
      for (int k = 0; k < p.pk_stages; ++k)
        if (armed[k]) mbar_wait(b.pk_full + 8 * k, armed_ph[k], &dummy, to);
    }
  } else if (warp >= kWarpMma0) {
    // ------------------------------------------------------------ MMA issuers
    // Issuer m owns the accumulators of segments m, m + kMmaWarps, ...; one
    // thread per warp, so independent accumulators are fed by parallel
    // instruction streams.
    const int m = warp - kWarpMma0;
    // a pair's MMAs issue from its even CTA, one issuer per segment
    if (lane == 0 && (!PAIR || (rank == 0 && m < kPairIssuers))) {
      int zs = 0;
      uint32_t zph = 0;
      long long nu = 0;
      bool ok = true;
      for (int it = it0; it < it1 && ok && !*abort_flag; it += it_step, ++nu) {
        const XItem item = item_at(p, it);
        const XProb pb = p.probs[item.prob];
        const XUnit *u = pb.units + item.tpl;
        const int n_seg = u->n_seg;
        static_assert(kMaxSegs == 2 * kMmaWarps, "two segments per issuer at most");
        // The (at most two) segments this issuer owns.  Their descriptors are
        // built once per item, for Z stage 0 and K slice 0, as 32-bit words:
        // a chunk in Z stage zs and K slice kk only adds (zs z_stage_bytes +
        // 32 kk) / 16 to the start-address field, so each MMA costs an add
        // or two and the instruction itself.  (One issuing thread shares its
        // SM sub-partition with four unpack warps; the fewer instructions it
        // needs per MMA, the sooner each MMA is issued.)
        const int n_mine = (m < n_seg) + (m + kMmaWarps < n_seg);
        uint32_t d_col[2], idesc[2], a_lo[2], b_lo[2], b_hi[2];
        const uint32_t z0 = smem_u32(z_buf), a_hi = sdesc_sw128_hi(1024u);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const XSeg &sgm = u->seg[j < n_mine ? m + kMmaWarps * j : 0];
          d_col[j] = tmem + (uint32_t)sgm.tmem_col;
          idesc[j] = idesc_e4m3_f32(PAIR ? 256 : 128, sgm.n);
          a_lo[j] = sdesc_sw128_lo(z0 + (uint32_t)sgm.a_zrow * 128u);
          b_lo[j] = sdesc_sw128_lo(z0 + (uint32_t)sgm.b_zrow * 128u);
          b_hi[j] = sdesc_sw128_hi((uint32_t)sgm.b_sbo);
        }
        if (nu > 0 &&
            !(PAIR ? mbar_wait_cluster(b.acc_empty, (uint32_t)((nu - 1) & 1), abort_flag, to)
                   : mbar_wait(b.acc_empty, (uint32_t)((nu - 1) & 1), abort_flag, to)))
          break;
        tc_fence_after();
        uint32_t acc0 = 0;  // the item's first MMA of each accumulator overwrites it
        StageWalk walk(pb, item.pk0);
        for (int k = 0; k < item.npk && ok; ++k, walk.next()) {
          const int nch = GRAM ? 1 : walk.chunks();
          for (int sub = 0; sub < nch; ++sub) {
            if (!(PAIR ? mbar_wait_cluster(b.z_full + 8 * zs, zph, abort_flag, to)
                       : mbar_wait(b.z_full + 8 * zs, zph, abort_flag, to))) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t zoff = ((uint32_t)zs * p.z_stage_bytes) >> 4;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              if (j >= n_mine) break;
              const uint32_t al = a_lo[j] + zoff, bl = b_lo[j] + zoff;
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                if (PAIR)
                  mma_f8_ss_w_pair(d_col[j], al + 2u * kk, a_hi, bl + 2u * kk, b_hi[j], idesc[j],
                                   kk ? 1u : acc0);
                else
                  mma_f8_ss_w(d_col[j], al + 2u * kk, a_hi, bl + 2u * kk, b_hi[j], idesc[j],
                              kk ? 1u : acc0);
              }
            }
            acc0 = 1;
            if (PAIR)
              mma_commit_pair(b.z_empty + 8 * zs, 3);  // both CTAs' operand stages
            else
              mma_commit(b.z_empty + 8 * zs);
            if (++zs == p.z_stages) { zs = 0; zph ^= 1u; }
          }
        }
        if (ok) {
          if (PAIR)
            mma_commit_pair(b.acc_full, 3);
          else
            mma_commit(b.acc_full);
        }
      }
      // all MMAs this thread issued complete before TMEM is released
      if (PAIR)
        mma_commit_pair(b.drain + 8 * m, 1);
      else
        mma_commit(b.drain + 8 * m);
      int dummy = 0;
      mbar_wait(b.drain + 8 * m, 0, &dummy, to);
    }
    if (PAIR && rank != 0 && m == 0 && lane == 0) {
      // The odd CTA's operand stages are announced to the even CTA's
      // issuers by this one thread: it waits for the local unpack warps'
      // arrivals, then makes a single cluster-scope release-arrive on the
      // even CTA's z_full (one cluster fence per chunk instead of one per
      // unpack warp).
      int zs = 0;
      uint32_t zph = 0;
      bool ok = true;
      for (int it = it0; it < it1 && ok && !*abort_flag; it += it_step) {
        const XItem item = item_at(p, it);
        const XProb pb = p.probs[item.prob];
        StageWalk walk(pb, item.pk0);
        for (int k = 0; k < item.npk && ok; ++k, walk.next()) {
          const int nch = walk.chunks();
          for (int sub = 0; sub < nch; ++sub) {
            if (!mbar_wait(b.z_full + 8 * zs, zph, abort_flag, to)) { ok = false; break; }
            mbar_arrive_cluster(b.z_full + 8 * zs, 0);
            if (++zs == p.z_stages) { zs = 0; zph ^= 1u; }
          }
        }
      }
    }
  } else if (warp < kUnpackWarps) {
    // ------------------------------------------------------------ unpack
    // The warps form two groups of kUnpackGroup, which decode the operand
    // chunks in turn (the even and the odd ones, counted over all items), so a
    // warp waits, fences and arrives once per two chunks, as a rule a packed
    // stage, and has all its loads of a chunk in flight together.  Taking turns
    // strictly, also past a block's odd last chunk, keeps a group at most two
    // chunks from its last wait on an operand stage: a parity wait then never
    // mistakes a stage's phase for the one two uses before.  (All warps on
    // every chunk spent half of their instructions on that hand-off: 3200 warp
    // instructions per chunk of 192 inputs.)  A region's inputs are a multiple
    // of kTileInputs, so every warp has the same number of 8-row groups: rows
    // 8 w + 64 k + 0..7 of the region, a lane one 16-sample group (lane / 8) of
    // one row (lane % 8); the 8 lanes of a quarter-warp take 8 consecutive
    // rows, so their swizzled 16-byte accesses fall on 8 different bank groups.
    const int grp = warp / kUnpackGroup, w8 = warp % kUnpackGroup;
    const int g = lane >> 3, sw = lane & 7;
    const int t_grp = 32 * w8 + lane;  // thread of the group
    // packed rows arrive 128B-swizzled: 16-byte chunk c of row r sits at
    // c ^ (r & 7); operand chunk `sub` of the stage is chunks 4 sub + g
    const uint32_t src_lane =
        (uint32_t)((8 * w8 + sw) * kPackedRowBytes + ((g ^ sw) << 4));
    // the lane's 32 operand bytes are 16-byte chunks 2 g and 2 g + 1 (Gram
    // form: a packed chunk's real and imaginary bytes go to the same chunk of
    // the two rows)
    const uint32_t dst_lane = (uint32_t)(sw * 128 + (((GRAM ? g : 2 * g) ^ sw) << 4));
    const uint32_t pk_s0 = smem_u32(pk_buf), z_s0 = smem_u32(z_buf);
    int s = 0, zs = 0;
    uint32_t ph = 0, zph = 0;
    bool ok = true;
    long long nu = 0;
    int turn = 0;  // the group that decodes the next chunk
    for (int it = it0; it < it1 && ok && !*abort_flag; it += it_step, ++nu) {
      const XItem item = item_at(p, it);
      const XProb pb = p.probs[item.prob];
      const XUnit *u = pb.units + item.tpl;
      const int n_reg = u->n_reg;
      // This thread's share of the operand sums: for each of its rows (F-
      // engine order: for each of its four inputs of a box), the sums of u
      // over the real parts (low half) and the imaginary parts (high half).
      uint32_t sums[2][TCN ? 8 : 4];
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int k = 0; k < (TCN ? 8 : 4); ++k) sums[r][k] = 0u;
      static_assert(kMaxFoldStages * 16 * 15 < 65536, "16-bit sums (Gram: 32 of half the stages)");
      int n_mine = 0;  // chunks this warp decoded
      // per-region constants (at most two regions of at most 256 inputs)
      uint32_t src_off[2], dst_off[2], dst_step[2];
      int n_k[2], kind[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const XRegion rg = u->reg[r < n_reg ? r : 0];
        kind[r] = rg.interleaved;
        n_k[r] = r < n_reg ? rg.n_in / kTileInputs : 0;
        src_off[r] = (uint32_t)rg.pk_off + (TCN ? 0u : src_lane);
        dst_step[r] = kind[r] ? 16384u : 8192u;  // 64 rows further on
        dst_off[r] = (uint32_t)rg.z_row * 128u +
                     (TCN ? 0u : (uint32_t)w8 * (dst_step[r] / kUnpackGroup) + dst_lane);
      }
      StageWalk walk(pb, item.pk0);
      for (int k = 0; k < item.npk; ++k, walk.next()) {
        const int nch = GRAM ? 1 : walk.chunks();
        const int sub = grp ^ turn;  // the group's chunk of this stage, if it has it
        turn ^= nch & 1;
        if (!mbar_wait(b.pk_full + 8 * s, ph, abort_flag, to)) { ok = false; break; }
        if (sub < nch) {
          ++n_mine;
          const int zm = zs + sub, zi = zm >= p.z_stages ? zm - p.z_stages : zm;
          const uint32_t zp = zm >= p.z_stages ? zph ^ 1u : zph;
          if (!mbar_wait(b.z_empty + 8 * zi, zp ^ 1u, abort_flag, to)) { ok = false; break; }
          const uint32_t pk_s = pk_s0 + (uint32_t)s * p.pk_stage_bytes;
          const uint32_t sub_x = GRAM || TCN ? 0u : 64u * (uint32_t)sub;  // chunks 4 on
          const uint32_t z_s = z_s0 + (uint32_t)zi * p.z_stage_bytes;
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            if (n_k[r] == 0) break;
            if constexpr (TCN && GRAM)
              unpack_gram_turned(pk_s + src_off[r], z_s + dst_off[r], n_k[r], t_grp, sums[r]);
            else if constexpr (GRAM)
              unpack_gram(pk_s + src_off[r], z_s + dst_off[r], n_k[r], sums[r]);
            else if constexpr (TCN)
              unpack_turned(pk_s + src_off[r], z_s + dst_off[r], kind[r], n_k[r], t_grp, sub,
                            sums[r]);
            else if (kind[r] == 1)
              unpack_rows<true>((pk_s + src_off[r]) ^ sub_x, z_s + dst_off[r], 16384u, n_k[r], sums[r]);
            else
              unpack_rows<false>((pk_s + src_off[r]) ^ sub_x, z_s + dst_off[r], dst_step[r], n_k[r], sums[r]);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(b.z_full + 8 * zi);
            mbar_arrive(b.pk_empty + 8 * s);
          }
        } else if (lane == 0) {
          mbar_arrive(b.pk_empty + 8 * s);  // not this group's, or a block's odd last chunk
        }
        if ((zs += nch) >= p.z_stages) { zs -= p.z_stages; zph ^= 1u; }
        if (++s == p.pk_stages) { s = 0; ph ^= 1u; }
      }
      if (!ok) break;
      // ---- the item's operand sums, for the epilogue, added up in a table
      // that it has cleared: entry = (Ua + Ub - 8 T, Ub - Ua) with Ua, Ub the
      // sums of u over the input's T real and imaginary parts (zero-filled
      // samples are u = 8, so they cancel)
      const uint32_t sum_ph = (uint32_t)(nu & 1) ^ 1u;
      if (!(PAIR ? mbar_wait_cluster(b.sum_empty, sum_ph, abort_flag, to)
                 : mbar_wait(b.sum_empty, sum_ph, abort_flag, to)))
        break;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int sum_row = u->reg[r < n_reg ? r : 0].sum_row;
#pragma unroll
        for (int k = 0; k < (TCN ? 8 : 4); ++k) {
          // whole warps: an 8-row group, or a quarter of a box, is in or out
          const int box = TCN ? 2 * (k >> 2) + (t_grp >> 7) : k;
          if (box >= n_k[r]) continue;
          int ua = (int)(sums[r][k] & 0xFFFFu), ub = (int)(sums[r][k] >> 16);
          if (!TCN) {
            ua += __shfl_xor_sync(0xffffffffu, ua, 8);
            ub += __shfl_xor_sync(0xffffffffu, ub, 8);
          }
          ua += __shfl_xor_sync(0xffffffffu, ua, 16);
          ub += __shfl_xor_sync(0xffffffffu, ub, 16);
          // normal order: the warp held all samples of a chunk of 8 rows; F-
          // engine order: a quarter of them (an eighth a half-warp) of 64 inputs
          if (lane < (TCN ? 16 : 8)) {
            int at;
            if (TCN) {
              const int i_rel = kTileInputs * box + 4 * (t_grp & 15) + (k & 3), gp = i_rel >> 3;
              at = 8 * gp + (((i_rel & 7) + (gp & 3)) & 7);  // by operand-row position
            } else {
              at = kTileInputs * k + 8 * w8 + sw;
            }
            const uint32_t addr =
                tab + 8u * (uint32_t)((int)rank * (p.sum_rows >> 1) + sum_row + at);
            constexpr int kSeen = (GRAM ? kPkSamples : kChunkSamples) / (TCN ? 4 : 1);
            const int vx = ua + ub - 8 * kSeen * n_mine;
            const int vy = ub - ua;
            reds32(addr, vx);
            reds32(addr + 4u, vy);
            if (PAIR) {
              red_cluster(addr, rank ^ 1u, vx);
              red_cluster(addr + 4u, rank ^ 1u, vy);
            }
          }
        }
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(b.sum_full);
        if (PAIR) mbar_arrive_cluster(b.sum_full, rank ^ 1u);
      }
    }
  } else if (warp < kWarpTma) {
    // ------------------------------------------------------------ epilogue
    // The warp's TMEM lane quarter holds 16 inputs, each a real row and, 8
    // lanes on, an imaginary one; each of the quarter's two warps folds 8 of
    // them.  A 16-lane load brings 16 columns of the 8 inputs, a thread
    // getting both parts of two column pairs of one input: the bias comes off
    // there, and the 8 x 16 complex values go through a 1 KB buffer so that
    // each atomic instruction adds 256 contiguous bytes of one row of the
    // integration buffer.  (Lane-per-row adds, 32 rows an instruction, made
    // four times the memory requests: the fold of a 192-input channel took 31
    // us.)
    const int q = warp & 3, h = (warp - kWarpEpi0) >> 2;
    const uint32_t ebuf = smem_u32(epi_mem) + (uint32_t)(warp - kWarpEpi0) * kEpiBufBytes;
    const int er = lane >> 2, ec = lane & 3;  // the thread's row and column pair as loaded
    // 16-byte chunk (4 k + ec) of buffer row er, swizzled by the row's parity
    const uint32_t est0 = ebuf + (uint32_t)(er * 128 + ((ec ^ ((er & 1) << 2)) << 4));
    const uint32_t est1 = ebuf + (uint32_t)(er * 128 + (((4 + ec) ^ ((er & 1) << 2)) << 4));
    // word `lane` of an even and of an odd row
    const uint32_t eld0 = ebuf + (uint32_t)(lane * 4);
    const uint32_t eld1 = ebuf + (uint32_t)((((lane >> 2) ^ 4) << 4) + (lane & 3) * 4);
    long long nu = 0;
    // failure-detection self-test: wait for a barrier that nothing completes;
    // the bounded wait gives up, raises the abort flag and every role winds
    // down (nothing is folded)
    if (p.selftest_never) mbar_wait(b.never, 0, abort_flag, to);
    for (int it = it0; it < it1; it += it_step, ++nu) {
      const XItem item = item_at(p, it);
      const XProb pb = p.probs[item.prob];
      const XUnit *u = pb.units + item.tpl;
      if (!mbar_wait(b.acc_full, (uint32_t)(nu & 1), abort_flag, to)) break;
      // once the kernel is winding down nothing more is folded: the
      // integration is void and is reported as such
      if (*abort_flag) break;
      tc_fence_after();
      if (!(PAIR ? mbar_wait_cluster(b.sum_full, (uint32_t)(nu & 1), abort_flag, to)
                 : mbar_wait(b.sum_full, (uint32_t)(nu & 1), abort_flag, to)))
        break;
      const uint32_t rank_off = PAIR ? (uint32_t)(p.sum_rows >> 1) * 8u : 0u;
      const long long acc_elems = (long long)pb.n_chan * pb.n_pairs * 2;
      const int n_seg = u->n_seg;
      for (int sg = 0; sg < n_seg; ++sg) {
        const XSeg sgm = u->seg[sg];
        const int rpc = GRAM ? sgm.ch_rows : 0;  // no other units hold several channels a tile
        // 8 inputs: group g of the tile.  In F-engine-order launches group
        // position l holds input (l - g) % 8 of the group, and column 8 G +
        // e the one at (e - G) % 8 (a row tile or column range starts at a
        // multiple of 64 inputs, so only g % 4 and G % 4 matter).
        const int g = 2 * q + h;
        const int i_tile = (rank ? sgm.row_in1 : sgm.row_in0) + 8 * g;
        // a tile of several channels: the 8 rows belong to channel block ci
        const int ci = rpc ? i_tile / rpc : 0;
        // a multi-channel unit's missing last channels (as unsigned, so that a
        // sum past 2^31 - 1 is past the last as well)
        const int c = (int)((uint32_t)item.chan + (uint32_t)sgm.chan_off + (uint32_t)ci);
        if ((uint32_t)c >= (uint32_t)pb.n_chan) continue;
        const int i0 = i_tile - ci * rpc;
        if (i0 >= pb.n_in) continue;
        int64_t *cacc = pb.acc + (long long)c * pb.n_pairs * 2;
        // the row's sums: the thread's row as loaded
        uint32_t p_i, m_i;
        lds64(tab + (rank ? rank_off : 0u) + 8u * (uint32_t)(sgm.a_sum + 8 * g + er), p_i, m_i);
        p_i += kMagicBits;
        m_i += kMagicBits;
        // the columns to fold: up to the 16 that hold the 8 rows' diagonal,
        // and of a multi-channel tile the rows' channel block only.  Column
        // blocks of a pair's segment are not in input order: all of them.
        // (Gram form: 16 inputs are 32 accumulator columns, 8 real ones and 8
        // imaginary ones in turn; cb counts inputs.)
        const int cb0 = rpc ? ci * rpc : 0;
        int cb1 = rpc ? cb0 + rpc : GRAM ? sgm.n >> 1 : sgm.n;
        if (!PAIR) cb1 = min(cb1, cb0 + ((i0 + 7 - (sgm.col_blk[0] + cb0 - ci * rpc)) & ~15) + 16);
        const uint32_t tm = tmem + ((uint32_t)(32 * q + 16 * h) << 16) + (uint32_t)sgm.tmem_col;
        uint32_t nxt[8], nxt2[8];
        __syncwarp();
        tmem_ld_16x256b_x2(tm + (uint32_t)(GRAM ? 2 * cb0 : cb0), nxt);
        if (GRAM) tmem_ld_16x256b_x2(tm + (uint32_t)(2 * cb0 + 16), nxt2);
        for (int cb = cb0; cb < cb1; cb += 16) {
          tmem_ld_wait();
          uint32_t v[8];
          if (GRAM) {
            // re re + im im, im re - re im: whole numbers below 2^24, exact
            auto f = [](uint32_t x) { return __uint_as_float(x); };
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const uint32_t *a = k ? nxt2 : nxt;
              v[4 * k] = __float_as_uint(f(a[0]) + f(a[6]));
              v[4 * k + 1] = __float_as_uint(f(a[1]) + f(a[7]));
              v[4 * k + 2] = __float_as_uint(f(a[2]) - f(a[4]));
              v[4 * k + 3] = __float_as_uint(f(a[3]) - f(a[5]));
            }
          } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = nxt[k];
          }
          // the next columns are on their way while these are folded
          if (cb + 16 < cb1) {
            tmem_ld_16x256b_x2(tm + (uint32_t)(GRAM ? 2 * cb + 32 : cb + 16), nxt);
            if (GRAM) tmem_ld_16x256b_x2(tm + (uint32_t)(2 * cb + 48), nxt2);
          }
          // input of the first column (one-CTA units: consecutive inputs)
          int j0 = sgm.col_blk[0] - ci * rpc + cb;
          if (PAIR) {
            if (cb >= 64) j0 = sgm.col_blk[1] + cb - 64;
            if (cb >= 128) j0 = sgm.col_blk[2] + cb - 128;
            if (cb >= 192) j0 = sgm.col_blk[3] + cb - 192;
            if (j0 > i0 + 7) continue;  // above the diagonal (uniform)
          }
          // the two column pairs' sums: of a pair's columns, the first half
          // is the even CTA's rows, the second the odd one's
          const int hc = PAIR && cb >= (sgm.n >> 1) ? 1 : 0;
          const uint32_t cs = tab + (hc ? rank_off : 0u) +
                              8u * (uint32_t)(sgm.b_sum + cb - hc * (sgm.n >> 1) + 2 * ec);
          const uint4 s0 = lds128(cs), s1 = lds128(cs + 64u);
          __syncwarp();  // the buffer's last values have been read
          sts128(est0, unbias(v[0], p_i + s0.x), unbias(v[2], m_i - s0.y),
                 unbias(v[1], p_i + s0.z), unbias(v[3], m_i - s0.w));
          sts128(est1, unbias(v[4], p_i + s1.x), unbias(v[6], m_i - s1.y),
                 unbias(v[5], p_i + s1.z), unbias(v[7], m_i - s1.w));
          __syncwarp();
          // lane w adds word w of each row: column w / 2, part w % 2
          const int jc = lane >> 1;
          const int j = TCN ? j0 + (jc & 8) + (((jc & 7) - (((cb + jc) >> 3) & 3)) & 7) : j0 + jc;
          int x[8];
#pragma unroll
          for (int r = 0; r < 8; ++r)
            x[r] = (int)(lds32((r & 1 ? eld1 : eld0) + (uint32_t)(r * 128)) - kMagicBits);
          // away from the diagonal and the last input every word counts
          const bool inside = j0 + 15 <= i0 && i0 + 7 < pb.n_in;
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const int i = i0 + (TCN ? ((r - (g & 3)) & 7) : r);
            if (inside || (i < pb.n_in && j <= i))
              acc_add(pb.acc, acc_elems, p.status,
                      cacc + (i * (i + 1) + 2 * j + (lane & 1)), x[r]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (PAIR && rank != 0)
          mbar_arrive_cluster(b.acc_empty, 0);
        else
          mbar_arrive(b.acc_empty);
        mbar_arrive(b.sum_read);
      }
      // once every epilogue warp has read the table it is cleared for the
      // next item
      if (!mbar_wait(b.sum_read, (uint32_t)(nu & 1), abort_flag, to)) break;
      for (int k = 32 * (warp - kWarpEpi0) + lane; k < p.sum_rows; k += 32 * kEpiWarps)
        sts64(tab + 8u * k, 0u, 0u);
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(b.sum_empty);
        if (PAIR) mbar_arrive_cluster(b.sum_empty, rank ^ 1u);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  // a pair's even CTA reads the odd one's operands and the odd one arrives on
  // the even one's barriers: neither leaves before both are done
  if (PAIR) cluster_sync();
  if (warp == kWarpMma0) {
    __syncwarp();
    tc_fence_after();
    if (PAIR)
      tmem_dealloc_pair(tmem, kTmemCols);
    else
      tmem_dealloc(tmem, kTmemCols);
  }
  if (threadIdx.x == 0 && *abort_flag) atomicOr(p.status, 1);
}

cudaError_t cmac_set_smem(int smem_bytes) {
  const void *kernels[] = {
      reinterpret_cast<const void *>(xengine_cmac_kernel<kMaxMaps, false, false, false>),
      reinterpret_cast<const void *>(xengine_cmac_kernel<kMaxMaps, true, false, false>),
      reinterpret_cast<const void *>(xengine_cmac_kernel<kMaxMaps, false, true, false>),
      reinterpret_cast<const void *>(xengine_cmac_kernel<kMaxMaps, true, true, false>),
      reinterpret_cast<const void *>(xengine_cmac_kernel<kMaxBatchMaps, false, false, false>),
      reinterpret_cast<const void *>(xengine_cmac_kernel<kMaxBatchMaps, false, true, false>),
      reinterpret_cast<const void *>(xengine_cmac_kernel<kMaxMaps, false, false, true>),
      reinterpret_cast<const void *>(xengine_cmac_kernel<kMaxMaps, true, false, true>),
      reinterpret_cast<const void *>(xengine_cmac_kernel<kMaxBatchMaps, false, false, true>)};
  for (const void *k : kernels) {
    cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_cmac(const XMaps &maps, const XParams &p, int grid, int smem_bytes,
                        cudaStream_t stream) {
  if (p.gram && p.tcn)
    xengine_cmac_kernel<kMaxMaps, true, false, true><<<grid, kThreads, smem_bytes, stream>>>(maps, p);
  else if (p.gram)
    xengine_cmac_kernel<kMaxMaps, false, false, true><<<grid, kThreads, smem_bytes, stream>>>(maps, p);
  else if (p.tcn)
    xengine_cmac_kernel<kMaxMaps, true, false, false><<<grid, kThreads, smem_bytes, stream>>>(maps, p);
  else
    xengine_cmac_kernel<kMaxMaps, false, false, false><<<grid, kThreads, smem_bytes, stream>>>(maps, p);
  return cudaGetLastError();
}

namespace {
// Launch configuration of the pair instance: clusters of two CTAs.
struct PairConfig {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  PairConfig(int clusters, int smem_bytes, cudaStream_t stream) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(2 * clusters);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = (size_t)smem_bytes;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
};
}  // namespace

cudaError_t launch_cmac_pair(const XMaps &maps, const XParams &p, int clusters, int smem_bytes,
                             cudaStream_t stream) {
  PairConfig c(clusters, smem_bytes, stream);
  if (p.tcn) return cudaLaunchKernelEx(&c.cfg, xengine_cmac_kernel<kMaxMaps, true, true, false>, maps, p);
  return cudaLaunchKernelEx(&c.cfg, xengine_cmac_kernel<kMaxMaps, false, true, false>, maps, p);
}

cudaError_t launch_cmac_batch_pair(const XBatchMaps &maps, const XParams &p, int clusters,
                                   int smem_bytes, cudaStream_t stream) {
  PairConfig c(clusters, smem_bytes, stream);
  return cudaLaunchKernelEx(&c.cfg, xengine_cmac_kernel<kMaxBatchMaps, false, true, false>, maps, p);
}

int cmac_pair_clusters(int smem_bytes) {
  PairConfig c(1, smem_bytes, nullptr);
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, xengine_cmac_kernel<kMaxMaps, false, true, false>, &c.cfg) ==
                 cudaSuccess
             ? n
             : 0;
}

int cmac_pair_clusters_batch(int smem_bytes) {
  PairConfig c(1, smem_bytes, nullptr);
  int n = 0;
  return cudaOccupancyMaxActiveClusters(&n, xengine_cmac_kernel<kMaxBatchMaps, false, true, false>,
                                        &c.cfg) == cudaSuccess
             ? n
             : 0;
}

cudaError_t launch_cmac_batch(const XBatchMaps &maps, const XParams &p, int grid, int smem_bytes,
                              cudaStream_t stream) {
  if (p.gram)
    xengine_cmac_kernel<kMaxBatchMaps, false, false, true>
        <<<grid, kThreads, smem_bytes, stream>>>(maps, p);
  else
    xengine_cmac_kernel<kMaxBatchMaps, false, false, false>
        <<<grid, kThreads, smem_bytes, stream>>>(maps, p);
  return cudaGetLastError();
}

}  // namespace xe
