// Shapes of the FP32 travel-time network's kernel (k_tt.cu) and the choice between
// its two forms.
#pragma once
#include <cstddef>
#include <cstdint>

namespace spider {

constexpr int kTP = 64;       // pairs per tile (wide form; the narrow form takes 32)
constexpr int kKC = 8;        // weight rows per staged chunk
constexpr int kStagesW = 3;   // chunks in flight
constexpr int kGroups = 8;    // partial sums over the hidden units: eight contiguous groups

// The narrow form: CTAs per SM (one, where two would leave a thread too few
// registers), and tiles of 32 pairs per SM up to which it is the faster form:
// 4864 pairs (one a SM) take 73 against 92 us at H = 128, 192 against 198 at 256;
// two a SM 55 against 71 us at H = 64, but 123 against 120 at H = 128; four a SM
// 44 against 66 us at H = 32.
constexpr int narrow_ctas(int H) { return H >= 64 ? 1 : 4; }
constexpr int narrow_tiles(int H) { return H >= 128 ? 1 : H >= 64 ? 2 : 4; }

// CTAs per SM of the wide form's persistent grid: no more than registers (64
// accumulators a thread, 128 registers) and shared memory (the activations of a tile
// and three weight chunks, 1 KB a CTA reserved beside them) hold at once, for tiles
// are dealt out by CTA and one that waits for a place runs its share alone (H = 32,
// 1,000,000 pairs: 804 us with eleven, 672 with ten)
constexpr int mlp_fp32_ctas(int H) { return H >= 256 ? 2 : H >= 128 ? 4 : H >= 64 ? 6 : 10; }

// Pairs of a step of n_b blocks, each of at most `nodes` pairs, in a catalog of P, at
// most.  (By the catalog's pairs alone, a small minibatch of a large catalog took the
// wide form and left SMs without a tile: a step of 1,000 pairs took 143 us at H = 64,
// 171 at 128 and 480 at 256, now 115, 151 and 270.)
constexpr int64_t step_pairs(int64_t P, int64_t n_b, int64_t nodes) { return n_b * nodes < P ? n_b * nodes : P; }

// whether a launch of at most n pairs takes the narrow form
constexpr bool narrow_form(int H, int64_t n, int num_sms) { return n <= (int64_t)32 * narrow_tiles(H) * num_sms; }

template <int H, bool WIDE>
struct Mlp32 {
  static constexpr int kPl = WIDE ? 2 : 1;           // pairs per lane
  static constexpr int kUw = WIDE ? 32 : 8;          // units per warp
  static constexpr int kTile = 32 * kPl;             // pairs per tile
  static constexpr int kThreads = H / kUw * 32;
  static constexpr int kChunkW = kKC * H;            // weights of a chunk
  static constexpr int kTotal = 6 * (H / kKC);       // chunks per tile
  static constexpr int kCtas = WIDE ? mlp_fp32_ctas(H) : narrow_ctas(H);
  static constexpr int kUpg = H / kGroups;           // units per partial sum
  static constexpr int kHold = WIDE ? 0 : H * kTile; // h4, kept for the sums of the narrow form
  // act, weight chunks, inputs, partial sums [kGroups][4][kTile], h4
  static constexpr size_t kSmem =
      (size_t)(H * kTile + kStagesW * kChunkW + 6 * kTile + kGroups * 4 * kTile + kHold) * sizeof(float);
};

}  // namespace spider
