// The GEMM's choice of a tile configuration: host code without CUDA, so that a
// CPU test can run it.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace qlin {

constexpr int kTileM = 128;         // rows of a CTA's tile (a pair tile: 256)
constexpr int kStageRowBytes = 128; // bytes of K per pipeline stage and row

enum class Tile { kPair, kSingle, kNarrow };   // 256 x 256, 128 x 128, 128 x 64
enum class GemmKind { kNvfp4, kFp8, k16 };     // k16: bf16 / fp16 operands

// What the epilogue does beside writing y.
enum class Epilogue { kPlain, kRequant, kAmax };

// Time of a launch in a tile configuration, in microseconds: a launch, then
// waves of tiles that each cost a start and end and their K stages.  Fitted
// to graph-replayed launches over M 16-4608, N 256-6144, K 256-3072 (operands
// in L2; rms error 5-9%).
struct TileCost {
  double launch, wave, stage;
  double us(int64_t tiles, int64_t slots, int64_t stages, double wave_extra) const {
    return launch +
           (double)((tiles + slots - 1) / slots) * (wave + wave_extra + (double)stages * stage);
  }
};

// Pair tiles when there are enough of them to fill the machine, else 128 x 128
// single-CTA tiles, or 128 x 64 when those would leave at least half the SMs
// idle -- unless the fitted times say that another configuration is at least 10%
// faster: mostly a last wave that is nearly empty (NVFP4 1000 x 3072 x 3072: 192
// single tiles on 152 SMs 10.4 us, 48 pair tiles 8.0) or a K too short for the
// pair tiles' start and end (NVFP4 4608 x 2560 x 256: pairs 7.8 us, single tiles
// 6.8).  The margin covers the fit's error.  Each configuration timed at 5934
// calls over M 16-18432, N 64-12288 and K 64-12288, far beyond the fit: the fit
// overrides the count in 795 of them, which take 0.81 of the time on average; ten
// are more than 5% slower for it, all with one or two waves or K = 64 (worst NVFP4
// 18432 x 1024 x 64: 10.4 -> 12.8 us).
inline Tile choose_tile(GemmKind kind, Epilogue epi, int64_t M, int64_t N, int64_t K,
                        int num_sms) {
  static const TileCost kCosts[3][3] = {
      {{2.5, 1.65, 0.24}, {2.7, 0.5, 0.29}, {2.7, 0.3, 0.26}},     // NVFP4
      {{3.3, 2.2, 0.265}, {2.7, 1.1, 0.205}, {2.8, 0.5, 0.175}},   // FP8
      {{3.0, 1.1, 0.275}, {2.6, 0.6, 0.18}, {2.6, 0.6, 0.18}}};    // bf16 / fp16
  const bool fp4 = kind == GemmKind::kNvfp4;
  // the fused re-quantization's 64-column groups need 128-column tiles, and no
  // 16-bit kernel has narrow ones
  const bool narrow_ok = epi != Epilogue::kRequant && kind != GemmKind::k16;
  const TileCost* cost = kCosts[(int)kind];
  const int64_t k_bytes = fp4 ? K / 2 : kind == GemmKind::k16 ? K * 2 : K;
  const int64_t stages = (k_bytes + kStageRowBytes - 1) / kStageRowBytes;
  const int64_t tiles_m = (M + kTileM - 1) / kTileM;
  const int64_t n128 = (N + 127) / 128, n256 = (N + 255) / 256;
  // An output amax costs single-CTA tiles more per wave (its reductions, and y
  // through the staging) and a pair tile more at its end: without these terms
  // short K chains took single tiles where pairs are faster (NVFP4 9216 x 3072 x 64:
  // 33.0 us, single tiles 37.6).
  const double wave_extra = epi == Epilogue::kAmax ? 0.2 : 0.0;
  double us[3] = {cost[0].us((tiles_m + 1) / 2 * n256, num_sms / 2, stages, 0.0),
                  cost[1].us(tiles_m * n128, num_sms, stages, wave_extra),
                  cost[2].us(tiles_m * ((N + 63) / 64), num_sms, stages, wave_extra)};
  // a pair tile's re-quantizing epilogue ends about this much later
  if (epi == Epilogue::kRequant) us[0] += fp4 ? 1.0 : 0.6;
  if (epi == Epilogue::kAmax) us[0] += 1.0;
  int pick = tiles_m * n256 >= num_sms ? 0 : narrow_ok && 2 * tiles_m * n128 <= num_sms ? 2 : 1;
  int best = pick;
  for (int t = 0; t < (narrow_ok ? 3 : 2); ++t)
    if (us[t] < us[best]) best = t;
  if (us[best] < 0.9 * us[pick]) pick = best;
  return static_cast<Tile>(pick);
}

}  // namespace qlin
