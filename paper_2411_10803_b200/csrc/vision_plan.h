// How the vision-encoding calls are laid out on the GPU: rules on sizes alone, host code without CUDA.
#pragma once

namespace mustdrop {

constexpr int kVisionWarps = 8;        // warps of a CTA of these kernels
constexpr int kMaxMergeCluster = 8;

// Vectors of each of a window's four tokens that a lane of the spatial merge has in flight, for rows of `vecs` vectors: a
// second one only where a row has more than the warp's 32 (62 images of 22 x 22 tokens x 96 channels: 13.2 us with one
// and four CTAs on an SM, 16.4 with two and three; 3 of 48 x 48 x 256: 26.6 and 28.5; 8 of 16 x 16 x 320: 7.7 both; 3 of
// 36 x 36 x 496: 20.5 and 19.0).
inline int merge_fly(int vecs) { return vecs > 32 ? 2 : 1; }

// CTAs per image of the spatial merge: the fewest rounds of windows (one per warp) in a row, over the waves of clusters
// that the GPU holds at once; of the same number of rounds the one with the fewest waves, whose CTAs start together; then
// the most CTAs.  resident[c]: clusters of c CTAs held at once.  (64 images of 144 windows: clusters of six, three full
// rounds in one wave; 42.7 -> 36.4 us together with the loads in flight.  96 of 36 windows x 512 channels: four CTAs,
// two rounds in one wave, 10.5 us; five, one round in each of two waves, 13.5.  One of 144 x 1024: eight CTAs 13.7 us,
// six, which take three rounds too, 15.1.)
inline int merge_cluster(int batch, int n_win, const int* resident) {
  int cluster = 1;
  long best = -1, best_waves = 0;
  for (int c = 1; c <= kMaxMergeCluster && (c - 1) * kVisionWarps < n_win; ++c) {
    const long waves = (batch + resident[c] - 1) / resident[c];
    const long rounds = waves * ((n_win + c * kVisionWarps - 1) / (c * kVisionWarps));
    if (best < 0 || rounds < best || (rounds == best && waves <= best_waves)) {
      best = rounds;
      best_waves = waves;
      cluster = c;
    }
  }
  return cluster;
}

// How the key set reads a token's row: a lane per vector of 16 bytes, or four or eight lanes with so many vectors each;
// steps of the warp's 32 lanes over its tokens in a trip; whether a trip's loads go out ahead of the trip before.
enum class KeyRows {
  kLanePerVector5,
  kLanePerVector3Ahead,
  kFour1x3Ahead,
  kFour1x5,
  kFour2x2,
  kFour2x2Ahead,
  kFour3x1Ahead,
  kEight2x2,
  kEight4x1Ahead,
};

// part: tokens of a warp's unit of work (half of a CTA's); ctas: CTAs of the call; sms: SMs of the device.
inline KeyRows key_rows(int head_dim, int part, int ctas, int sms) {
  const bool full = 2L * ctas >= 5L * sms;   // five CTAs and more on two SMs
  if (head_dim <= 32) {
    // Four lanes with a vector each, three steps ahead: 24 tokens a trip.  Up to 16 dimensions that leaves two or three of
    // four lanes without a vector, which shows where a unit is more than one trip or, with one vector to a row, the
    // batch fills the GPU (us for a lane per vector, four lanes; 12 images of 1936 tokens, 12 x 8: 14.2, 22.6; x 16: 17.8,
    // 22.5; 24 of 576, 16 x 8: 14.1, 18.1; 96 of 256, 12 x 8: 18.2, 19.2; but x 16: 21.0, 19.4; 4 of 300, 12 x 16: 10.1,
    // 9.2; x 8: 9.3, 9.2).
    if (head_dim <= 16 && (part > 24 || (head_dim <= 8 && full))) return KeyRows::kLanePerVector5;
    // Units that take two trips of three steps but one of five: five at once (24 images of 576 tokens, 16 x 24: 18.1 us
    // with three ahead, 15.8 with five, 17.5 with a lane per vector; 40 of 400, 16 x 32: 18.0, 15.6, 17.2; longer ones are
    // as fast with three ahead: 3 of 700, 16 x 32: 12.2, 13.7, 15.7).
    return part > 24 && part <= 40 ? KeyRows::kFour1x5 : KeyRows::kFour1x3Ahead;
  }
  if (head_dim <= 64) {
    // Four lanes with two vectors each, two steps at once; the form with loads ahead spills (16 x 64 dimensions, us for five
    // steps of a lane per vector, two steps of four lanes ahead, at once: 24 images of 576 tokens: 25.1, 24.5, 20.2; 24 of 320:
    // 17.3, 19.3, 15.8; 39 of 1731, 12 heads: 47.3, 38.2, 33.7; 40 of 320: 17.9, 20.1, 16.8).
    if (!full) return KeyRows::kFour2x2;
    // Where the batch fills the GPU and the merge's writes are still on their way, whole lines of 128 bytes in flight all
    // the time are ahead: a lane per vector, three steps ahead (merge and key set of 64 images of 576 tokens x 1024 channels,
    // 16 x 64 dimensions: 69.3 us for two steps ahead, 75 at once, 65.5; 48 images: 62.5, 61.9, 57.0; 44, where it is not
    // full: 54.3, 52.6, 55.6).  But for units of one trip of four lanes (64 of 256 tokens: 43.2, 45.3, 45.3), and of one trip of
    // five steps that three would take two for (96 of 320 tokens, the key set alone: 32.2 us with five steps, 34.0).
    if (part <= 16) return KeyRows::kFour2x2Ahead;
    return part <= 20 ? KeyRows::kLanePerVector5 : KeyRows::kLanePerVector3Ahead;
  }
  if (head_dim <= 96) return KeyRows::kFour3x1Ahead;
  // Eight lanes.  A lane per vector with three steps ahead made calls of 20 to 120 tokens a unit slower than five steps
  // without had been (us for five steps, three ahead, eight lanes: 4 images of 300 tokens, 12 x 104 dimensions: 14.9, 16.2,
  // 11.2; 15 of 2007, 16 x 104: 103, 114, 66; 64 of 576, 16 x 128: 44.8, 45.0, 42.8; 64 of 576, 16 x 160: 80.9, 82.5, 51.7;
  // 12 of 1936, 12 x 256: 136, 118, 86).
  return head_dim <= 128 ? KeyRows::kEight2x2 : KeyRows::kEight4x1Ahead;
}

}  // namespace mustdrop
