// xe_sched.cu -- triangle covers, shared-memory stage layout and the balanced
// split of a launch into per-CTA item runs (host code only).
#include "xe_sched.h"

#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <utility>

namespace xe {

namespace {

int round_up(int v, int m) { return (v + m - 1) / m * m; }

void add_seg(XUnit &u, int a_zrow, int b_zrow, int b_sbo, int n, int row_in0, int col_in0) {
  XSeg &s = u.seg[u.n_seg];
  int col = 0;
  for (int k = 0; k < u.n_seg; ++k) col += u.seg[k].n;
  s.a_zrow = a_zrow;
  s.b_zrow = b_zrow;
  s.b_sbo = b_sbo;
  s.n = n;
  s.tmem_col = col;
  s.row_in0 = row_in0;
  s.row_in1 = row_in0;
  for (int b = 0; b < 4; ++b) s.col_blk[b] = col_in0 + 64 * b;
  u.n_seg++;
  u.work += n;
}

void add_reg(XUnit &u, int in_lo, int n_in, int interleaved) {
  XRegion &r = u.reg[u.n_reg];
  r.in_lo = in_lo;
  r.in_lo1 = in_lo;
  r.n_in = n_in;
  r.interleaved = interleaved;
  r.z_row = u.z_rows;
  r.pk_off = u.pk_bytes;
  r.sum_row = u.n_sum;
  u.z_rows += interleaved ? 2 * n_in : n_in;
  u.n_sum += n_in;
  u.pk_bytes += n_in * kPackedRowBytes;
  u.n_reg++;
}

// Entry of the table of operand sums that belongs to Z row z of unit u (the
// row of an 8-row group of A rows).
int sum_entry(const XUnit &u, int z) {
  for (int r = 0; r < u.n_reg; ++r) {
    const XRegion &g = u.reg[r];
    const int step = g.interleaved ? 2 : 1;
    if (z >= g.z_row && z < g.z_row + step * g.n_in) return g.sum_row + (z - g.z_row) / step;
  }
  return 0;
}

XUnit empty_unit() {
  XUnit u;
  std::memset(&u, 0, sizeof(u));
  u.n_chan = 1;
  return u;
}

}  // namespace

// Entries of the table of operand sums for a finished unit's segments.
static void set_sums(XUnit &u) {
  for (int s = 0; s < u.n_seg; ++s) {
    u.seg[s].a_sum = sum_entry(u, u.seg[s].a_zrow);
    u.seg[s].b_sum = sum_entry(u, u.seg[s].b_zrow);
  }
}

static int gram_units(int N, XUnit *units, int tiles) {
  const int n16 = round_up(N, 16);
  XUnit &u = units[0] = empty_unit();
  u.gram = 1;
  if (N <= kTileInputs) {
    // tiles of one channel each, or of 64 / n16 channels (ch_rows)
    const int cpt = N <= 32 ? kTileInputs / n16 : 1;
    u.n_chan = tiles * cpt;
    for (int r = 0; r < tiles; ++r) {
      add_reg(u, 0, kTileInputs, 1);
      u.reg[r].chan_off = r * cpt;
    }
    for (int r = 0; r < tiles; ++r) {
      add_seg(u, u.reg[r].z_row, u.reg[r].z_row, 1024, N <= 32 ? 2 * kTileInputs : 2 * n16, 0, 0);
      u.seg[r].chan_off = r * cpt;
      u.seg[r].ch_rows = N <= 32 ? n16 : 0;
    }
  } else {
    // two row tiles of one channel, at most 128 + 256 columns
    add_reg(u, 0, 2 * kTileInputs, 1);
    add_seg(u, 128, 0, 1024, 2 * n16, kTileInputs, 0);
    add_seg(u, 0, 0, 1024, 2 * kTileInputs, 0, 0);
  }
  set_sums(u);
  return 1;
}

// Tiles of 64 inputs (rows) cover the lower triangle strip by strip: row tile
// t needs columns [0, min(64 (t + 1), N)).  Within a unit, columns are staged
// once per chunk and shared by all its row tiles.
int window_units(int N, XUnit *units, int tiles) {
  if (N <= kGramInputs) return gram_units(N, units, tiles);
  const int n16 = round_up(N, 16);
  const int n_rt = (N + kTileInputs - 1) / kTileInputs;
  int n_units = 0;
  // units of consecutive row tiles, largest strip first, each as many as
  // fit 512 TMEM columns: a unit's lowest tile then bounds the inputs that
  // are only its columns, and those need no Q rows
  for (int t_max = n_rt - 1; t_max >= 0;) {
    int t_min = t_max + 1, used = 0;
    while (t_min > 0) {
      const int n = std::min(kTileInputs * t_min, n16);  // tile t_min - 1
      if (used + n > kTmemCols) break;
      used += n;
      --t_min;
    }
    XUnit &u = units[n_units++] = empty_unit();
    // inputs below the unit's lowest row tile are only its columns: plain
    // rows, with MMAs of their own.  (In the interleaved layout, Q slots
    // empty, one MMA spans both, but a stage takes 64 KB, only two fit, and
    // the unpack and the issuers wait for each other: 256 inputs 1354 us a
    // launch against 1294, and 1118 with the split's costs set right.)
    const int own = kTileInputs * t_min;
    if (t_min > 0) add_reg(u, 0, own, 0);
    add_reg(u, own, kTileInputs * (t_max + 1 - t_min), 1);
    const int z_own = u.reg[u.n_reg - 1].z_row;
    for (int t = t_max; t >= t_min; --t) {
      const int a_zrow = z_own + 128 * (t - t_min);
      if (t_min > 0) add_seg(u, a_zrow, 0, 1024, own, kTileInputs * t, 0);
      add_seg(u, a_zrow, z_own, 2048, std::min(kTileInputs * (t + 1), n16) - own,
              kTileInputs * t, own);
    }
    t_max = t_min - 1;
  }
  for (int k = 0; k < n_units; ++k) set_sums(units[k]);
  return n_units;
}

std::vector<XUnit> build_schedule(int N, int cover) {
  std::vector<XUnit> units;
  const int n16 = round_up(N, 16);
  const int n_rt = (N + kTileInputs - 1) / kTileInputs;
  if (N <= 256 && cover == kCoverWindow) {
    XUnit w[kMaxWindowUnits];
    units.assign(w, w + window_units(N, w));
  } else if (N <= 256 && cover == kCoverStrips) {
    for (int t = n_rt - 1; t >= 0; --t) {
      XUnit u = empty_unit();
      add_reg(u, 0, kTileInputs * (t + 1), 1);
      add_seg(u, 128 * t, 0, 2048, std::min(kTileInputs * (t + 1), n16), kTileInputs * t, 0);
      units.push_back(u);
    }
  } else if (N > 256 && cover == kCoverQuads) {
    // CTA pairs, blocks of 256 rows [R, R + 256) against 256 columns
    // [P, P + 256), P <= R, in four row tiles T0..T3 of 64 inputs.
    //  - Below the diagonal (P < R) the even CTA owns T0 and T1, the odd one
    //    T2 and T3; their B rows are a plain region, P .. P + 127 on the even
    //    CTA and P + 128 .. on the odd one.  Two N = 256 MMAs.
    //  - On the diagonal (P = R) the even CTA owns T0 and T3, the odd one T1
    //    and T2, and each CTA's own A rows are its B rows: the MMA of T0 and
    //    T1 (N = 128) takes the first 64 B rows of each CTA, columns T0 T1;
    //    that of T3 and T2 (N = 256) all of them, columns T0 T3 T1 T2.  That
    //    issues 3/4 of the work of two N = 256 MMAs over T0 T1 | T2 T3.
    for (int R = 0; R < N; R += 2 * kPairRows) {
      for (int P = 0; P <= R; P += 2 * kPairRows) {
        XUnit u = empty_unit();
        u.pair_rows = kPairRows;
        if (P < R) {
          add_reg(u, R, kPairRows, 1);
          u.reg[0].in_lo1 = R + kPairRows;
          add_reg(u, P, kPairRows, 0);
          u.reg[1].in_lo1 = P + kPairRows;
          const int bz = u.reg[1].z_row;
          for (int t = 0; t < 2; ++t) {
            add_seg(u, 128 * t, bz, 1024, 2 * kPairRows, R + kTileInputs * t, P);
            u.seg[t].row_in1 = R + kPairRows + kTileInputs * t;
          }
        } else {
          const int T = kTileInputs;
          add_reg(u, R, T, 1);  // even: T0, odd: T1
          u.reg[0].in_lo1 = R + T;
          add_reg(u, R + 3 * T, T, 1);  // even: T3, odd: T2
          u.reg[1].in_lo1 = R + 2 * T;
          add_seg(u, 0, 0, 2048, 2 * T, R, R);
          u.seg[0].row_in1 = R + T;
          u.seg[0].col_blk[1] = R + T;
          add_seg(u, 128, 0, 2048, 4 * T, R + 3 * T, R);
          u.seg[1].row_in1 = R + 2 * T;
          u.seg[1].col_blk[1] = R + 3 * T;
          u.seg[1].col_blk[2] = R + T;
          u.seg[1].col_blk[3] = R + 2 * T;
        }
        units.push_back(u);
      }
    }
  } else {
    // pairs of row tiles (2m, 2m+1) against W-column pieces of their strip;
    // above 256 inputs, where a piece's columns are staged beside 128 rows,
    // 192 columns (256 would leave no shared memory for the operand sums)
    const int W = N > 256 ? 192 : 256;
    for (int m = 0; 2 * m < n_rt; ++m) {
      const int t0 = 2 * m;
      const bool two = t0 + 1 < n_rt;
      const int row_lo = kTileInputs * t0;
      const int kd = row_lo / W;  // piece holding the diagonal
      for (int k = 0; k <= kd; ++k) {
        XUnit u = empty_unit();
        if (k < kd) {
          add_reg(u, row_lo, two ? 128 : 64, 1);
          add_reg(u, W * k, W, 0);
          const int bz = u.reg[1].z_row;
          add_seg(u, 0, bz, 1024, W, row_lo, W * k);
          if (two) add_seg(u, 128, bz, 1024, W, row_lo + 64, W * k);
        } else {
          const int lo = W * k;
          const int hi = row_lo + (two ? 128 : 64);
          // inputs lo .. row_lo - 1 are only columns here: no Q rows
          if (row_lo > lo) add_reg(u, lo, row_lo - lo, 2);
          add_reg(u, row_lo, hi - row_lo, 1);
          const int a0 = 2 * (row_lo - lo);
          add_seg(u, a0, 0, 2048, std::min(row_lo + 64, n16) - lo, row_lo, lo);
          if (two) add_seg(u, a0 + 128, 0, 2048, std::min(row_lo + 128, n16) - lo, row_lo + 64, lo);
        }
        units.push_back(u);
      }
    }
  }
  std::stable_sort(units.begin(), units.end(),
                   [](const XUnit &a, const XUnit &b) { return a.work > b.work; });
  for (XUnit &u : units) set_sums(u);
  // the unpack handles regions of at most kMaxRegionInputs inputs (every
  // cover above satisfies this; an empty schedule reports a violation)
  for (const XUnit &u : units)
    for (int r = 0; r < u.n_reg; ++r)
      if (u.reg[r].n_in > kMaxRegionInputs) return {};
  return units;
}

int tile_ch_rows(const std::vector<XUnit> &units) {
  for (const XUnit &u : units)
    for (int s = 0; s < u.n_seg; ++s)
      if (u.seg[s].ch_rows) return u.seg[s].ch_rows;
  return kTileInputs;
}

XUnit tm_unit(int n_in) {
  const TmGeom G = tm_geom(n_in);
  XUnit u = empty_unit();
  add_reg(u, 0, kTileInputs * G.n_rt, 1);
  u.work = G.acc_cols;
  return u;
}

int launch_cover(int n_in) {
  if (n_in <= 256) return kCoverWindow;
  const char *e = std::getenv("CORR_CMAC_KERNEL");
  const bool one_cta = e && std::strcmp(e, "smem") == 0;
  return n_in > kPairInputs && !one_cta ? kCoverQuads : kCoverPairs;
}

bool stage_layout(const std::vector<const std::vector<XUnit> *> &unit_sets, int smem_optin,
                  int max_z, StageLayout *out) {
  int max_zr = 0, max_pk = 0, max_sum = 0;
  for (const auto *set : unit_sets)
    for (const XUnit &u : *set) {
      max_zr = std::max(max_zr, u.z_rows);
      max_pk = std::max(max_pk, u.pk_bytes);
      max_sum = std::max(max_sum, (u.pair_rows ? 2 : 1) * u.n_sum);
    }
  return stage_layout(max_zr, max_pk, max_sum, smem_optin, max_z, out);
}

bool stage_layout(int max_zr, int max_pk, int max_sum, int smem_optin, int max_z,
                  StageLayout *out) {
  StageLayout L;
  L.sum_rows = max_sum;
  L.z_stage_bytes = (uint32_t)round_up(max_zr * 128, 1024);
  L.pk_stage_bytes = (uint32_t)round_up(max_pk, 1024);  // swizzled TMA destination
  const int fixed = 1024 /* alignment slack */ + kBarrierBytes + kEpiWarps * kEpiBufBytes +
                    max_sum * kSumBytesPerInput;
  static_assert(8 * (2 * kMaxPkStages + 2 * kMaxZStages + 2 + kMmaWarps + 1 + 3) + 16 <=
                    kBarrierBytes,
                "barrier area");
  const int avail = smem_optin - fixed;
  const int zb = (int)L.z_stage_bytes, pb = (int)L.pk_stage_bytes;
  const int zcap = std::min(max_z, kMaxZStages);
  // Operand stages first (three beside three packed stages, else three
  // beside two, else two beside three or two), then a fourth, then packed
  // stages (bytes in flight from HBM), and both up to their caps while they
  // fit.  (Six packed stages before the fourth operand stage: 64 inputs 626 us
  // a launch against 612.)
  int zs, ps;
  if (3 * zb + 3 * pb <= avail && zcap >= 3) {
    zs = 3;
    ps = 3;
  } else if (3 * zb + 2 * pb <= avail && zcap >= 3) {
    // (the CTA-pair units: a third operand stage hides the peer's arrivals)
    zs = 3;
    ps = 2;
  } else if (2 * zb + 3 * pb <= avail) {
    zs = 2;
    ps = 3;
  } else if (2 * zb + 2 * pb <= avail) {
    zs = 2;
    ps = 2;
  } else {
    return false;
  }
  auto grow = [&](int &v, int cap, int bytes) {
    while (v < cap && zs * zb + ps * pb + bytes <= avail) ++v;
  };
  grow(zs, std::min(4, zcap), zb);
  grow(ps, kMaxPkStages, pb);
  grow(zs, zcap, zb);
  L.z_stages = zs;
  L.pk_stages = ps;
  L.smem_bytes = fixed + zs * zb + ps * pb;
  // one CTA per SM: the kernel holds all 512 TMEM columns
  L.smem_bytes = std::max(L.smem_bytes, smem_optin / 2 + 1024);
  L.smem_bytes = std::min(L.smem_bytes, smem_optin);
  *out = L;
  return true;
}

int chunk_cost(const XUnit &u) {
  int mma = 0, rows = 0;
  for (int s = 0; s < u.n_seg; ++s) mma += 4 * ((u.pair_rows ? 54 : 24) + u.seg[s].n / 2);
  for (int r = 0; r < u.n_reg; ++r) rows += (u.reg[r].interleaved == 1 ? 2 : 1) * u.reg[r].n_in;
  const int cost = std::max(mma, 450 + 12 * rows / 5);
  return u.gram ? cost / 2 : cost;  // its rows and MMAs hold 128 samples
}

// Modelled cycles of the busiest CTA of a split.
static long long busiest(const std::vector<ProbWork> &probs, const std::vector<XItem> &items,
                         const std::vector<int> &cta_first) {
  long long most = 0;
  for (size_t b = 0; b + 1 < cta_first.size(); ++b) {
    long long sum = 0;
    for (int k = cta_first[b]; k < cta_first[b + 1]; ++k) {
      const XUnit &u = (*probs[items[k].prob].units)[items[k].tpl];
      sum += (long long)kChunksPerPk * items[k].npk * chunk_cost(u) + kFold * u.work;
    }
    most = std::max(most, sum);
  }
  return most;
}

int build_items_filled(const std::vector<ProbWork> &probs, int grid, std::vector<XItem> &items,
                       std::vector<int> &cta_first) {
  int used = build_items(probs, grid, items, cta_first);
  if (used <= 0) return used;
  long long best = busiest(probs, items, cta_first);
  // with many items per CTA the runs are balanced and finer pieces only add
  // folds
  if ((int)items.size() > 4 * grid) return used;
  std::vector<XItem> it;
  std::vector<int> first;
  auto keep_if_better = [&]() {
    const long long t = busiest(probs, it, first);
    if (t >= best) return;
    best = t;
    items.swap(it);
    cta_first.swap(first);
  };
  int npk = 0, nseg = 1;
  for (const ProbWork &pr : probs)
    npk = std::max(npk, (pr.block_len + kPkSamples - 1) / kPkSamples * pr.n_blocks);
  // finer cuts of the runs, where a unit is long enough for two pieces (the
  // search is host time of every corr_create: at 2048 inputs x 7 channels x 16
  // samples it took 0.5 of 1.0 ms to find the same split three times)
  for (int min_split = 8; min_split >= 2; min_split /= 2) {
    if (npk < 2 * min_split) continue;
    build_items(probs, grid, it, first, min_split);
    keep_if_better();
  }
  // every unit in n equal pieces, dealt round the CTAs (where a fold costs more
  // than a CTA's share of the work, no run is cut): the n of the shortest
  // modelled run, rounds of the costliest unit's pieces
  long long n_units = 0, fold = 0, work = 0;
  for (const ProbWork &pr : probs) {
    for (const XUnit &u : *pr.units) {
      n_units += channel_units(pr.n_chan, u.n_chan);
      fold = std::max(fold, kFold * u.work);
      work = std::max(work, (long long)kChunksPerPk * chunk_cost(u));
    }
  }
  nseg = (npk + kMaxFoldStages - 1) / kMaxFoldStages;
  int best_n = 0;
  for (int n = nseg; n <= std::min(npk, 64 * nseg); ++n) {
    const long long t = (n_units * n + grid - 1) / grid * ((npk + n - 1) / n * work + fold);
    if (t < best) best = t, best_n = n;
    if (n_units * n >= 2LL * grid) break;
  }
  if (best_n == 0) return (int)cta_first.size() - 1;
  it.clear();
  for (size_t p = 0; p < probs.size(); ++p) {
    const ProbWork &pr = probs[p];
    const int pk = (pr.block_len + kPkSamples - 1) / kPkSamples * pr.n_blocks;
    const int n = std::min(pk, std::max(best_n, (pk + kMaxFoldStages - 1) / kMaxFoldStages));
    for (int t = 0; t < (int)pr.units->size(); ++t)
      for (int w = 0, step = (*pr.units)[t].n_chan; w < channel_units(pr.n_chan, step); ++w)
        for (int k = 0; k < n; ++k) {
          const int lo = (int)((long long)pk * k / n), hi = (int)((long long)pk * (k + 1) / n);
          it.push_back({(int)p, t, w * step, lo, hi - lo});
        }
  }
  used = std::min(grid, (int)it.size());
  items.clear();
  cta_first.assign(1, 0);
  for (int b = 0; b < used; ++b) {
    for (size_t k = b; k < it.size(); k += used) items.push_back(it[k]);
    cta_first.push_back((int)items.size());
  }
  return used;
}

int tune_channels(const std::vector<std::vector<XUnit>> &schedules, int n_sm) {
  int most = 1;
  for (const std::vector<XUnit> &units : schedules)
    for (const XUnit &u : units) most = std::max(most, u.n_chan);
  return n_sm * most;
}

int build_items(const std::vector<ProbWork> &probs, int grid, std::vector<XItem> &items,
                std::vector<int> &cta_first, int min_split_pk, int max_item_pk) {
  items.clear();
  cta_first.clear();
  // Cost model, in SM cycles: chunk_cost per 64-sample chunk of a unit, and
  // kFold per accumulator column for its fold.
  struct PW {
    int cpb, ppb, npk, nseg;  // nseg: fold-window segments of a unit's stages
  };
  if (max_item_pk < 1) max_item_pk = 1;
  std::vector<PW> pw(probs.size());
  long long total = 0;
  for (size_t p = 0; p < probs.size(); ++p) {
    const ProbWork &pr = probs[p];
    pw[p].cpb = (pr.block_len + kChunkSamples - 1) / kChunkSamples;
    pw[p].ppb = (pr.block_len + kPkSamples - 1) / kPkSamples;
    pw[p].npk = pw[p].ppb * pr.n_blocks;
    pw[p].nseg = (pw[p].npk + max_item_pk - 1) / max_item_pk;
    for (const XUnit &u : *pr.units)
      total += (long long)channel_units(pr.n_chan, u.n_chan) *
               ((long long)pw[p].cpb * pr.n_blocks * chunk_cost(u) + kFold * u.work * pw[p].nseg);
  }
  if (total == 0 || grid <= 0) {
    cta_first.push_back(0);
    return 0;
  }
  // cost of stages [a, b) of a unit that costs `per_chunk` a chunk
  auto range_cost = [&](size_t p, int a, int b, int per_chunk) {
    // all stages but a block's last one hold kChunksPerPk chunks
    const int ppb = pw[p].ppb, short_by = kChunksPerPk * ppb - pw[p].cpb;
    const long long chunks =
        (long long)kChunksPerPk * (b - a) - (long long)short_by * (b / ppb - a / ppb);
    return chunks * per_chunk;
  };
  // The templates of a channel read the same inputs.  Where there are many, its
  // units run at the same time, so that the inputs come from L2 (2048 inputs
  // on CTA pairs: contiguous runs spread the CTAs over all channels, and the
  // loads alone, from HBM, took 4.6 of 4.7 ms against 3.0 ms from L2): units go
  // channel by channel to the CTA that is free first, and one that would
  // overrun the mean load is cut there.  Up to kRunTemplates one-CTA templates
  // contiguous runs are faster, every CTA having about the same mix of units
  // (384 inputs 619 / 752 us, 512 1095 / 1175, 768 1129 / 1220, 896 1523 /
  // 1567, 1152 1333 / 1306; 1280 inputs on pairs 1558 / 1381).
  constexpr size_t kRunTemplates = 20;
  bool shared_inputs = false;
  for (const ProbWork &pr : probs)
    for (const XUnit &u : *pr.units)
      shared_inputs = shared_inputs || u.pair_rows || pr.units->size() > kRunTemplates;
  if (shared_inputs) {
    std::vector<std::vector<XItem>> runs(grid);
    typedef std::pair<long long, int> Load;  // modelled cost so far, CTA
    // a heap whose top is the CTA that is free first; a deal raises the top's
    // cost and lets it sink (a priority queue's pop and push, and the costs
    // worked out anew for each unit, made up most of a large context's creation)
    std::vector<Load> heap;
    for (int k = 0; k < grid; ++k) heap.push_back({0, k});
    auto before = [](const Load &a, const Load &b) {  // without a branch
      return (a.first < b.first) | ((a.first == b.first) & (a.second < b.second));
    };
    auto sink_top = [&]() {
      const Load x = heap[0];
      size_t at = 0;
      for (size_t c = 1; c < heap.size(); c = 2 * at + 1) {
        c += (c + 1 < heap.size()) && before(heap[c + 1], heap[c]);
        if (before(x, heap[c])) break;
        heap[at] = heap[c];
        at = c;
      }
      heap[at] = x;
    };
    long long mean = (total + grid - 1) / grid;
    auto deal_next = [&](size_t p, int t, int c, int pk, int npk, long long per, long long fold) {
      while (pk < npk) {
        Load &l = heap[0];
        const long long room = mean - l.first - fold;
        int n = npk - pk;
        if (per * n > room) {
          const int fit = (int)std::max<long long>(0, room / per);
          if (fit >= min_split_pk && n - fit >= min_split_pk) {
            n = fit;
            total += fold;  // the rest of the unit is folded once more
            mean = (total + grid - 1) / grid;
          }
        }
        runs[l.second].push_back({(int)p, t, c, pk, n});
        l.first += per * n + fold;
        sink_top();
        pk += n;
      }
    };
    for (size_t p = 0; p < probs.size(); ++p) {
      const std::vector<XUnit> &us = *probs[p].units;
      const long long npk_total = pw[p].npk;
      const int nseg = pw[p].nseg;
      int step = 1;  // channels of a unit (the same for all templates)
      std::vector<long long> per, fold;  // cost of a template's stage and of its fold
      for (const XUnit &u : us) {
        step = std::max(step, u.n_chan);
        per.push_back((long long)kChunksPerPk * chunk_cost(u));
        fold.push_back(kFold * u.work);
      }
      for (int w = 0; w < channel_units(probs[p].n_chan, step); ++w)
        for (int sg = 0; sg < nseg; ++sg)
          for (int t = 0; t < (int)us.size(); ++t)
            deal_next(p, t, w * step, (int)(npk_total * sg / nseg),
                      (int)(npk_total * (sg + 1) / nseg), per[t], fold[t]);
    }
    cta_first.push_back(0);
    for (const std::vector<XItem> &run : runs) {
      if (run.empty()) continue;
      items.insert(items.end(), run.begin(), run.end());
      cta_first.push_back((int)items.size());
    }
    return (int)cta_first.size() - 1;
  }
  long long remaining = total, load = 0;
  int cta = 0;
  long long target = (remaining + grid - 1) / grid;
  cta_first.push_back(0);
  auto close_cta = [&]() {
    remaining -= load;
    load = 0;
    ++cta;
    cta_first.push_back((int)items.size());
    if (cta < grid) target = (remaining + (grid - cta) - 1) / (grid - cta);
  };
  // deals the stages [pk, npk) of unit (p, t, c) over the CTAs
  auto deal = [&](size_t p, int t, int c, int pk, int npk) {
    const XUnit &u = (*probs[p].units)[t];
    const int per_chunk = chunk_cost(u);
    const long long fold = kFold * u.work;
    while (pk < npk) {
      if (cta == grid - 1) {  // the last CTA takes everything left
        const long long cost = range_cost(p, pk, npk, per_chunk) + fold;
        items.push_back({(int)p, t, c, pk, npk - pk});
        load += cost;
        pk = npk;
        continue;
      }
      const long long rest = range_cost(p, pk, npk, per_chunk) + fold;
      if (load + rest <= target) {
        items.push_back({(int)p, t, c, pk, npk - pk});
        load += rest;
        pk = npk;
        if (load >= target) close_cta();
        continue;
      }
      // the rest overflows this CTA: take the stages that fit, if that
      // leaves pieces of at least min_split_pk stages on both sides
      int n = 0;
      const long long room = target - load - fold;
      if (room > 0) {
        const long long per = (long long)kChunksPerPk * per_chunk;
        n = (int)std::min<long long>(npk - pk, room / per);
        while (n > 0 && range_cost(p, pk, pk + n, per_chunk) > room) --n;
      }
      if (n >= min_split_pk && npk - pk - n >= min_split_pk) {
        items.push_back({(int)p, t, c, pk, n});
        load += range_cost(p, pk, pk + n, per_chunk) + fold;
        remaining += fold;  // the rest of the unit is folded once more
        pk += n;
        close_cta();
      } else if (load == 0 || 2 * (load + rest - target) < rest) {
        // no useful split: the whole rest goes here when this CTA is
        // empty or when most of the rest fits
        items.push_back({(int)p, t, c, pk, npk - pk});
        load += rest;
        pk = npk;
        close_cta();
      } else {
        close_cta();
      }
    }
  };
  for (size_t p = 0; p < probs.size(); ++p) {
    const long long npk_total = pw[p].npk;
    const int nseg = pw[p].nseg;
    for (int t = 0; t < (int)probs[p].units->size(); ++t)
      for (int w = 0, step = (*probs[p].units)[t].n_chan;
           w < channel_units(probs[p].n_chan, step); ++w)
        // fold-window segment sg: stages [npk sg / nseg, npk (sg + 1) / nseg)
        for (int sg = 0; sg < nseg; ++sg)
          deal(p, t, w * step, (int)(npk_total * sg / nseg), (int)(npk_total * (sg + 1) / nseg));
  }
  if (load > 0 || (int)cta_first.size() == 1) close_cta();
  // drop trailing empty CTAs
  while (cta_first.size() > 2 && cta_first[cta_first.size() - 2] == cta_first.back())
    cta_first.pop_back();
  return (int)cta_first.size() - 1;
}

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Looked up once; threads that come first together all find the same address.
EncodeTiledFn get_encode_fn() {
  static std::atomic<EncodeTiledFn> known{nullptr};
  EncodeTiledFn fn = known.load(std::memory_order_acquire);
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
    if (fn) known.store(fn, std::memory_order_release);
  }
  return fn;
}

}  // namespace

bool encode_block_map(const void *base, int block_len, int n_in, int n_chan, int pitch, void *map,
                      int ch_rows) {
  static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
  EncodeTiledFn enc = get_encode_fn();
  if (!enc) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)block_len, (cuuint64_t)n_in, (cuuint64_t)n_chan};
  const cuuint64_t strides[2] = {(cuuint64_t)pitch, (cuuint64_t)pitch * (cuuint64_t)n_in};
  if (ch_rows != 16 && ch_rows != 32 && ch_rows != kTileInputs) return false;
  const cuuint32_t box[3] = {(cuuint32_t)kPkSamples, (cuuint32_t)ch_rows,
                             (cuuint32_t)(kTileInputs / ch_rows)};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(static_cast<CUtensorMap *>(map), CU_TENSOR_MAP_DATA_TYPE_UINT8, 3,
                   const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B,
                   // a row's next stage comes along into L2
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool encode_block_map_tcn(const void *base, int block_len, int n_in, int n_chan, void *map,
                          int ch_rows) {
  EncodeTiledFn enc = get_encode_fn();
  if (!enc || n_in % 16 != 0) return false;
  if (ch_rows != 16 && ch_rows != 32 && ch_rows != kTileInputs) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)n_in, (cuuint64_t)n_chan, (cuuint64_t)block_len};
  const cuuint64_t strides[2] = {(cuuint64_t)n_in, (cuuint64_t)n_in * (cuuint64_t)n_chan};
  // ch_rows inputs of 64 / ch_rows channels: each sample of the box is still
  // 64 bytes, channel-major, as the tile's rows are
  const cuuint32_t box[3] = {(cuuint32_t)ch_rows, (cuuint32_t)(kTileInputs / ch_rows),
                             (cuuint32_t)kPkSamples};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(static_cast<CUtensorMap *>(map), CU_TENSOR_MAP_DATA_TYPE_UINT8, 3,
                   const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace xe
