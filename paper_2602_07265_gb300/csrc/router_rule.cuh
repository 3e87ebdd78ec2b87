// Which router a batch takes, host side.
#pragma once

namespace xs {

// The tensor cores' costs about 9 us whatever the batch; the CUDA cores' grows
// with the work.  Below 64 tokens the latter always wins; for narrow layers (d
// < kRouterSplitMinD) up to B N d of about kRouterFmas, as long as the logits
// are few enough: its blocks of 8 tokens x 4 experts have a fixed cost, which
// is most of it for small d.  Layer forward on GB300, plain top-k, tensor |
// CUDA cores, us:
//   d = 2048: N = 64, B = 150 (20 M) 67.3 | 64.3, 250 (33 M) 68.5 | 67.6, 350
//   (46 M) 68.9 | 69.4; N = 256, B = 64 (34 M) 101.2 | 98.9, 100 (52 M) 92.7 | 93.2
//   d = 3072, N = 128: B = 64 (25 M) 88.4 | 86.9, 128 (50 M) 85.1 | 86.1
//   by B N, in thousands, F = 128:
//   d = 128: N = 128, B = 256 (33) 30.9 | 32.2, 512 (66) 33.9 | 40.2, 1984 (254)
//   47.7 | 82.1; N = 32, B = 1024 (33) 37.7 | 38.9, 2048 (66) 43.3 | 49.3
//   d = 256: N = 128, B = 128 (16) 31.2 | 29.9, 256 (33) 33.1 | 33.9, 992 (127)
//   41.9 | 57.0; N = 32, B = 512 (16) 34.9 | 34.3, 1024 (33) 38.3 | 39.6
//   d = 512: N = 32, B = 512 (16) 37.3 | 35.5, 1024 (33) 40.7 | 41.0; N = 128, B =
//   128 (16) 36.3 | 34.3, 256 (33) 38.2 | 38.9, 496 (63) 42.2 | 46.0
//   d = 1024: N = 32, B = 512 (16) 43.7 | 40.5, 992 (32) 45.8 | 45.4
// (The CUDA cores' sums are the more exact ones: largest relative error of a
// score against 64 bits 1.0 to 1.4e-6, the tensor cores' 3.0 to 3.5e-6.)
constexpr int kRouterTcMinB = 64;
constexpr long long kRouterFmas = 32ll << 20;
constexpr long long kRouterLogits = 24 << 10;
constexpr int kRouterSplitMinD = 4096;
constexpr int kRouterSplitMaxD = 16384;

inline bool router_on_tensor_cores(int B, int N, int d) {
  const long long logits = static_cast<long long>(B) * N;
  return B >= kRouterTcMinB && (d >= kRouterSplitMinD || logits * d > kRouterFmas || logits > kRouterLogits);
}

}  // namespace xs
