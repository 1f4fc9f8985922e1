// Launch plans: the default rule for a shape (tiles, group length, split count), the
// checks a plan must pass, and the buffer layout quantities that depend on the plan.  A
// plan depends on the shape only, never on the data or the load.
#include <algorithm>
#include <string>

#include "rsim_internal.h"

namespace rsim {

namespace {
// The FP32 tier runs on the tensor cores from frames of kFp32TensorPixels pixels on: hi + lo
// FP16 operands, three products, at most kFp32Group chunks in an accumulator, FP32 sums of
// those.  It is closer to FP64 than the FP32 sum on the CUDA cores (over 364 frames of 128 to
// 65,536 pixels 0.6 of its error in the middle, 1.13 at most, with strengths of one phase) and
// faster (relative error and time, tensor / CUDA cores, log-normal strengths):
//   512 x 512 pixels, V = 8,  N_s = 512, L = 256   5.4e-7 / 1.79e-6   2517 / 29280 us
//   256 x 256,        V = 12, N_s = 256, L = 128   4.1e-7 / 1.29e-6    272 / 2816 us
//   128 x 128,        V = 8,  N_s = 256, L = 128   3.1e-7 / 6.8e-7      81 / 492 us
//   32 x 32,          V = 8,  N_s = 64,  L = 32    2.8e-7 / 4.8e-7      39 / 73 us
//   16 x 8,           V = 2,  N_s = 64,  L = 16    2.8e-7 / 3.6e-7      31 / 42 us
// Frames of a few chunks take as long either way (5 x 3 pixels: 25-29 / 26 us).  With 0 to 30%
// of background every one of 118 frames from 128 pixels on was as fast or faster (0.99 to 2.3
// times); with 90% the CUDA-core sum's fewer launches win below some 10,000 pixels (25 / 35 us),
// but the valid count is not known when the form is chosen.
constexpr int kFp32Group = 2;
constexpr int64_t kFp32TensorPixels = 128;
}  // namespace

int tile_nt(int L) { return L >= 128 ? 128 : ((L + 7) / 8) * 8; }

int64_t tensor_split_stride(int V, int Ns, int L, int nt) {
  const int64_t mtiles = ((int64_t)V * Ns + 127) / 128;
  return mtiles * ((L + nt - 1) / nt) * 128 * nt;
}

bool uses_partial(int tier, int64_t P, int splits, int group) {
  if (tier == RSIM_TIER_NUFFT) return false;
  if (splits > 1) return true;
  if (tier == RSIM_TIER_FP32 || tier == kTierFp32Tensor) return false;  // the sums stay in registers
  const int64_t chunks = (P + kChunkPx - 1) / kChunkPx;
  return chunks > group;
}

int group_chunks(int tier) {
  if (tier == kTierFp32Tensor) return kFp32Group;
  return split_tier(tier) ? 40 : 96;
}

// The split tiers' 2e-5 bar leaves room for the round-toward-zero bias of at most 40
// chunks (480 accumulating MMAs, a relative shrink of about 1e-5); the plain 16-bit tiers
// (1e-2) allow 384 chunks (1536 MMAs, about 3e-5).
int group_chunks_max(int tier) {
  if (tier == kTierFp32Tensor) return kFp32Group;
  return split_tier(tier) ? 40 : 384;
}

bool fp32_on_tensor_cores(int64_t P) { return P >= kFp32TensorPixels; }

int units_per_split(int tier, int V, int Ns, int L, int tile_n) {
  if (tier == RSIM_TIER_FP32) return V * ((Ns + tile_n - 1) / tile_n) * ((L + kDirectTileL - 1) / kDirectTileL);
  const int64_t rows = (int64_t)V * Ns;
  const int64_t trows = tier == kTierFp32Tensor ? 256 : 128;  // a pair of CTAs takes two row tiles
  return (int)(((rows + trows - 1) / trows) * ((L + tile_n - 1) / tile_n));
}

int default_splits(int tier, int V, int Ns, int L, int tile_n, int64_t P, int num_sms) {
  if (tier == RSIM_TIER_NUFFT) return 1;
  const int tiles = units_per_split(tier, V, Ns, L, tile_n);
  const int64_t chunks = (P + kChunkPx - 1) / kChunkPx;
  // keep at least 8 chunks (256 pixels) per split
  int64_t smax = chunks / 8 > 0 ? chunks / 8 : 1;
  if (smax > kMaxSplits) smax = kMaxSplits;
  if (tier == RSIM_TIER_FP32) {
    // FP32 accumulation: at most 8192 pixels per split, so that the running sum of
    // random-phase terms keeps a relative rounding error of a few 1e-6 (the splits are
    // then added with compensated sums); above that, the split count that fills whole
    // waves of two resident CTAs per SM best
    const int64_t smin = std::min<int64_t>(std::max<int64_t>((P + 8191) / 8192, 1), kMaxSplits);
    const int64_t slots = 2ll * num_sms;
    double best = -1.0;
    int64_t bs = smin;
    for (int64_t s = smin; s <= std::max(smin, smax); ++s) {
      const int64_t units = (int64_t)tiles * s;
      const int64_t waves = (units + slots - 1) / slots;
      const double eff = (double)units / (double)(waves * slots) - 0.001 * s;
      if (eff > best + 1e-9) {
        best = eff;
        bs = s;
      }
    }
    return (int)bs;
  }
  // tensor tiers: one persistent CTA (or half a pair) per SM takes equal units in turn; pick
  // the split count whose unit count fills whole rounds best, with a small cost per split for
  // the partial sums it adds.  That cost has to stay below the SMs' share of one unit, or a
  // frame of one tile is not split at all (0.01 against 1 / 152: one CTA works, 8 to 50 times
  // as long).  On pairs a unit's share is 1 / 76, and 0.01 is the better line there (64 frames
  // of 12 tiles: 6 splits instead of 19, 10.40 ms against 11.21)
  const bool on_pairs = tier == kTierFp32Tensor;
  const int slots = std::max(on_pairs ? num_sms / 2 : num_sms, 1);
  const double per_split = std::min(on_pairs ? 0.01 : 0.003, 0.75 / slots);
  double best = -1.0;
  int bs = 1;
  for (int s = 1; s <= smax; ++s) {
    const int64_t units = (int64_t)tiles * s;
    const int64_t rounds = (units + slots - 1) / slots;
    const double eff = (double)units / (double)(rounds * slots) - per_split * s;
    if (eff > best + 1e-9) {
      best = eff;
      bs = s;
    }
  }
  return bs;
}

void resolve_tile(int tier, const Consts& k, rsim_plan* p) {
  if (tier == RSIM_TIER_FP32) {
    if (p->tile_n == 0) p->tile_n = kDirectTileN;
    p->group_chunks = 0;
  } else if (tensor_tier(tier)) {
    if (p->tile_n == 0) p->tile_n = tile_nt(k.L);
    if (p->group_chunks == 0) p->group_chunks = group_chunks(tier);
  } else {
    p->tile_n = 0;
    p->group_chunks = 0;
  }
  p->chunk_px = kChunkPx;
}

rsim_plan default_plan(int tier, const Consts& k, int64_t P, int num_sms) {
  rsim_plan p{};
  resolve_tile(tier, k, &p);
  p.splits = default_splits(tier, k.V, k.Ns, k.L, p.tile_n, P, num_sms);
  return p;
}

std::string plan_problem(int tier, const Consts& k, const rsim_plan& p) {
  if (p.splits < 1 || p.splits > kMaxSplits) return "plan splits must be in 1..64";
  if (p.grid < 0) return "plan grid must be >= 0";
  if (p.variant != 0) return "plan variant must be 0";
  if (tier == RSIM_TIER_FP32) {
    if (p.tile_n != 0 && p.tile_n != 64 && p.tile_n != 128) return "FP32 tile_n must be 64 or 128";
  } else if (tensor_tier(tier)) {
    const int lmax = std::max(8, (k.L + 7) / 8 * 8);
    if (p.tile_n != 0 && (p.tile_n < 8 || p.tile_n > 128 || p.tile_n % 8 != 0 || p.tile_n > lmax))
      return "tensor-core tile_n must be a multiple of 8 in 8..min(128, L rounded up to 8)";
    if (p.group_chunks < 0 || p.group_chunks > group_chunks_max(tier))
      return "group_chunks must be in 1.." + std::to_string(group_chunks_max(tier)) + " for this tier";
  }
  return std::string();
}

}  // namespace rsim
