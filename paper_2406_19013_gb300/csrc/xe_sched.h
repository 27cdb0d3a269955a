// xe_sched.h -- host-side scheduling of the CMAC kernel: the cover of the lower
// triangle by MMA tiles (templates) and the split of a launch's work into
// per-CTA runs of items of about equal cost.  Not part of the public ABI.
#pragma once
#include <cstdint>
#include <vector>

#include "xe_internal.h"

namespace xe {

// Cover variants of the triangle (the autotuner chooses between them).
enum Cover {
  // N <= 256: one staged window of all inputs per unit; consecutive row
  // tiles' strips, largest first, packed into units of <= 512 TMEM columns.
  // Up to kGramInputs inputs in the Gram form.
  kCoverWindow = 0,
  // N <= 256: one unit per row tile t, staging inputs [0, 64 (t + 1)) only.
  kCoverStrips = 1,
  // any N: pairs of row tiles against 256-column pieces of their strip,
  // 192-column pieces for N > 256 (the only one-CTA cover there).
  kCoverPairs = 2,
  // N > 256, CTA pairs: blocks of 256 rows (four row tiles, two per CTA)
  // against 256-column pieces of their strip, each piece's B rows split
  // between the two CTAs (units with pair_rows = kPairRows).
  kCoverQuads = 3,
};

// Largest input count whose units run on one CTA each by default; above it CTA
// pairs.  A pair's MMAs share their column operand, so each SM unpacks fewer
// rows per product, but its 256-row blocks pad more and its two CTAs wait for
// each other.  CMAC launches, one CTA / pairs: 300 inputs 0.75 / 1.16 ms, 512
// 1.15 / 1.25 ms (128 channels, 2 blocks of 8192 samples); 32 channels, 4
// blocks of 4096: 1152 inputs 1.30 / 1.39 ms, 1280 1.56 / 1.42, 2048 3.62 /
// 3.21.
constexpr int kPairInputs = 1152;

// The cover that launches of n_in inputs run (contexts, batches without the
// autotuner, the host views): CTA pairs above kPairInputs, unless
// CORR_CMAC_KERNEL=smem in the environment asks for one-CTA units.
int launch_cover(int n_in);

// Templates of the cover, heaviest first.  kCoverWindow and kCoverStrips
// fall back to kCoverPairs above 256 inputs, kCoverQuads at 256 and below.
std::vector<XUnit> build_schedule(int n_in, int cover);

// The window cover's templates, heaviest first, into units[kMaxWindowUnits]
// (n_in <= 256; allocates nothing).  Returns their number; all of them cover
// the same number of channels.
constexpr int kMaxWindowUnits = 4;
// tiles: 64-row tiles of a unit of at most 64 inputs (1 or 2), each with its
// own channels.
int window_units(int n_in, XUnit *units, int tiles = 2);

// Up to kGramInputs inputs the window cover's units are of the Gram form: the
// same triangle with half of the operand bytes.  A tile's 128 rows are the real
// and the imaginary rows of 64 inputs, 128 samples to a 128-byte row (against
// [re, im] and [im, -re] rows of 64 samples), and D holds re re, re im, im re
// and im im products, which the epilogue adds up.  No negated rows are decoded
// or stored, a stage is one hand-off instead of two, and the MMAs are twice as
// wide; but an input takes two accumulator columns, so a channel of more than
// 128 inputs does not fit the 512 TMEM columns.
constexpr int kGramInputs = 128;

// The unit that the item split models for the TMEM-operand kernel (up to
// kTmMaxInputs inputs): the operand rows that its unpack decodes, two for each
// staged input, and its accumulator columns.  No launch reads it.
XUnit tm_unit(int n_in);

// Modelled cycles of one 64-sample chunk of a unit: the unpack of its operand
// rows, with the hand-off of the chunk (measured at 300 to 512 inputs: 1047
// cycles for 192 rows written, 1065 for 256, 1260 for 320, 1448 for 384, 1527
// for 448), or its MMAs if they take longer (four K slices of each segment, on
// shared-memory operands 57 cycles at N = 64, 122 at 192, 155 at 256, and 182
// for a CTA pair's M = 256, N = 256).  Fitted where two operand stages fit and
// the unpack binds; with three or more the two overlap better (192 inputs: 1371
// modelled, 1100 to 1130 measured, folds included, bound by the MMAs), and the
// TMA stream that binds Gram units is not modelled (532 modelled; 666 measured
// at 128 inputs, 693 at 64, 755 at 16).  The splits use the costs of a launch's
// units against each other and against kFold, which weighs a third too little
// where the model is a third too high.
int chunk_cost(const XUnit &u);
// Modelled cycles of a unit's fold per accumulator column (measured: 384
// columns in about 20 000 cycles).
constexpr long long kFold = 50;

// Shared-memory layout of a launch whose units are `units`.
struct StageLayout {
  int z_stages, pk_stages;
  uint32_t z_stage_bytes, pk_stage_bytes;
  int sum_rows;  // entries of a table of operand sums
  int smem_bytes;
};
// The stages that fit `smem_optin`: three operand stages beside three or two
// packed ones, or else two beside three or two; then a fourth operand stage,
// packed stages up to kMaxPkStages and operand stages up to max_z, while they
// fit.  Returns false if not even 2 + 2 stages fit.
bool stage_layout(const std::vector<const std::vector<XUnit> *> &unit_sets, int smem_optin,
                  int max_z, StageLayout *out);

// The same for units of at most max_zr operand rows, max_pk packed bytes and
// max_sum entries of operand sums (allocates nothing).
bool stage_layout(int max_zr, int max_pk, int max_sum, int smem_optin, int max_z,
                  StageLayout *out);

// Units of per_unit channels that n_chan channels take (no int on the way
// exceeds n_chan: unit w starts at channel w per_unit < n_chan).
constexpr int channel_units(int n_chan, int per_unit) { return (n_chan - 1) / per_unit + 1; }

// One problem as the item builder sees it.
struct ProbWork {
  const std::vector<XUnit> *units;
  int n_chan;
  int block_len;
  int n_blocks;  // blocks in the launch
};

// Packed stages one item may integrate before its fold: 32768 samples.  The
// biased operands are integers u in [0, 15], so a sample adds at most
// 2 x 15^2 = 450 to an accumulator (in units of 2^-18) and 32768 of them stay
// below 2^24: every fp32 partial is exact.
constexpr int kMaxFoldStages = 32768 / kPkSamples;
static_assert(2LL * 15 * 15 * kMaxFoldStages * kPkSamples < (1LL << 24), "exact fp32 partials");

// Cuts every unit (problem, template, channel) into items and deals them to at
// most `grid` CTAs, in contiguous runs, or, where many templates or CTA pairs
// share a channel's inputs, channel by channel to the CTA that is free first.
// Each CTA receives about the same modelled cost: chunk_cost for every chunk of
// its items, plus kFold per accumulator column for the fold of each.  A unit is
// split only at 128-sample stage boundaries and only into pieces of at least
// min_split_pk stages; first it is cut into equal segments of at most
// max_item_pk stages (the fold window), which every item stays inside.
// Fills items and cta_first (size used_grid + 1) and returns used_grid.
int build_items(const std::vector<ProbWork> &probs, int grid, std::vector<XItem> &items,
                std::vector<int> &cta_first, int min_split_pk = 16,
                int max_item_pk = kMaxFoldStages);

// As build_items, for a launch that is to fill the SMs: where the units are few,
// finer cuts and equal pieces of every unit are tried as well and the split
// whose busiest CTA is modelled shortest is taken (16 inputs x 64 channels x
// 2048 samples: 8 units of 16 stages ran on 8 CTAs, and run on 128).
int build_items_filled(const std::vector<ProbWork> &probs, int grid, std::vector<XItem> &items,
                       std::vector<int> &cta_first);

// Channels of a problem on which schedules are timed against each other: a
// unit for every SM, whichever schedule's units hold the most channels (with
// as many channels as SMs, 16 inputs' Gram units ran on 19 of 152).
int tune_channels(const std::vector<std::vector<XUnit>> &schedules, int n_sm);

// The TMA descriptor of one block, uint8 [n_chan][n_in][row pitch], 3-D
// (time, input, channel) with boxes of 128 samples x ch_rows inputs x
// 64 / ch_rows channels (64 rows in all), 128B-swizzled.  ch_rows is 64
// except for schedules whose tiles hold several channels (16 or 32, see
// XSeg::ch_rows and tile_ch_rows).  `map` receives 128 bytes.  Returns false
// if the driver's encoder is unavailable or rejects the arguments.
bool encode_block_map(const void *base, int block_len, int n_in, int n_chan, int pitch, void *map,
                      int ch_rows = kTileInputs);

// Inputs per channel in a 64-row tile of a schedule's units: 16 or 32 when
// its tiles hold several channels, else 64.
int tile_ch_rows(const std::vector<XUnit> &units);

// The TMA descriptor of one block in F-engine order, uint8 [block_len][n_chan]
// [n_in], 3-D (input, channel, time) with 64-input x 1-channel x 128-sample
// boxes, no swizzle (each box lands as [128 samples][64 inputs]).  The
// channel and time strides must be multiples of 16 bytes: n_in % 16 == 0.
bool encode_block_map_tcn(const void *base, int block_len, int n_in, int n_chan, void *map,
                          int ch_rows = kTileInputs);

}  // namespace xe
