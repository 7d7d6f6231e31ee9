// Block width nb of lu_factor(nb = 0), by factorization kind and size:
// the fastest candidate of an offline sweep of whole solves (factor +
// solve or refinement) on the benchmarks' seeded matrices.  Generated by
//   python -m paper_2202_13995_gb300.tune
// on NVIDIA GB300; times in ms (best of the repetitions after a warm-up).
#pragma once

namespace gb {

// kind: 0 FP64 (certified split update), 1 FP64 (split tensor-core update),
// 2 BF16 / FP16 mixed, 3 FP32.  The first entry of the kind whose nmax
// is at least n applies.
struct NbEntry {
  int kind, nmax, nb;
};

constexpr NbEntry kNbTable[] = {
    {0, 800, 32},  // f64, measured at n = 600: nb 32: 1.727, nb 64: 1.832, nb 96: 1.822, nb 128: 1.822, nb 192: 2.119, nb 256: 2.215
    {0, 1280, 64},  // f64, measured at n = 1023: nb 32: 3.372, nb 64: 3.378, nb 96: 3.405, nb 128: 3.399, nb 192: 3.890, nb 256: 4.052
    {0, 3072, 128},  // f64, measured at n = 2048: nb 32: 11.491, nb 64: 8.497, nb 96: 8.119, nb 128: 7.863, nb 192: 8.313, nb 256: 8.813
    {0, 4608, 128},  // f64, measured at n = 4096: nb 32: 54.039, nb 64: 24.168, nb 96: 21.382, nb 128: 19.882, nb 192: 19.895, nb 256: 20.440
    {0, 7168, 192},  // f64, measured at n = 6000: nb 32: 145.503, nb 64: 50.987, nb 96: 42.636, nb 128: 37.990, nb 192: 36.308, nb 256: 36.872
    {0, 12288, 256},  // f64, measured at n = 8192: nb 32: 340.574, nb 64: 101.188, nb 96: 80.685, nb 128: 69.635, nb 192: 63.104, nb 256: 62.336
    {0, 24576, 256},  // f64, measured at n = 16384: nb 32: 2521.305, nb 64: 608.801, nb 96: 447.020, nb 128: 361.227, nb 192: 289.931, nb 256: 260.948
    {0, 1073741824, 256},  // f64, measured at n = 32768: not measured: n = 32768 keeps the smaller size's choice
    {1, 1280, 128},  // f64_split, measured at n = 1024: nb 64: 4.817, nb 128: 4.150, nb 192: 4.416, nb 256: 4.354
    {1, 3072, 128},  // f64_split, measured at n = 2048: nb 64: 10.953, nb 128: 9.130, nb 192: 9.128, nb 256: 9.207
    {1, 4608, 256},  // f64_split, measured at n = 4096: nb 64: 28.511, nb 128: 21.894, nb 192: 20.868, nb 256: 20.433
    {1, 7168, 256},  // f64_split, measured at n = 7001: nb 64: 77.134, nb 128: 53.242, nb 192: 47.253, nb 256: 45.692
    {1, 12288, 256},  // f64_split, measured at n = 8192: nb 64: 107.476, nb 128: 71.496, nb 192: 61.973, nb 256: 58.585
    {1, 24576, 256},  // f64_split, measured at n = 16384: nb 64: 607.516, nb 128: 353.454, nb 192: 274.128, nb 256: 237.480
    {1, 1073741824, 256},  // f64_split, measured at n = 32768: nb 64: 4066.466, nb 128: 2244.717, nb 192: 1653.813, nb 256: 1410.500
    {2, 800, 128},  // mixed, measured at n = 600: nb 64: 1.076, nb 128: 0.868, nb 192: 0.895, nb 256: 0.859, nb 384: 0.847
    {2, 1280, 256},  // mixed, measured at n = 1024: nb 64: 1.488, nb 128: 1.267, nb 192: 1.192, nb 256: 1.121, nb 384: 1.169
    {2, 3072, 256},  // mixed, measured at n = 2048: nb 64: 2.814, nb 128: 2.167, nb 192: 2.183, nb 256: 2.117, nb 384: 2.275
    {2, 4608, 256},  // mixed, measured at n = 4096: nb 64: 5.862, nb 128: 4.535, nb 192: 4.551, nb 256: 4.417, nb 384: 4.636
    {2, 7168, 256},  // mixed, measured at n = 6000: nb 64: 9.361, nb 128: 7.218, nb 192: 7.065, nb 256: 6.793, nb 384: 7.189
    {2, 12288, 256},  // mixed, measured at n = 8192: nb 64: 14.909, nb 128: 10.821, nb 192: 10.198, nb 256: 9.608, nb 384: 10.458
    {2, 24576, 256},  // mixed, measured at n = 16384: nb 64: 57.702, nb 128: 35.933, nb 192: 30.219, nb 256: 27.199, nb 384: 28.869
    {2, 1073741824, 256},  // mixed, measured at n = 32768: nb 64: 299.866, nb 128: 171.840, nb 256: 127.095, nb 384: 127.630, nb 512: 136.121
    {3, 800, 128},  // f32, measured at n = 600: nb 64: 0.874, nb 128: 0.750, nb 192: 0.806, nb 256: 0.794
    {3, 1280, 128},  // f32, measured at n = 1024: nb 64: 1.321, nb 128: 1.126, nb 192: 1.187, nb 256: 1.163
    {3, 3072, 128},  // f32, measured at n = 2048: nb 64: 2.628, nb 128: 2.247, nb 192: 2.322, nb 256: 2.321
    {3, 4608, 128},  // f32, measured at n = 4096: nb 64: 6.874, nb 128: 6.089, nb 192: 6.238, nb 256: 6.220
    {3, 12288, 128},  // f32, measured at n = 8192: nb 64: 27.834, nb 128: 24.786, nb 192: 24.857, nb 256: 24.671
    {3, 24576, 256},  // f32, measured at n = 16384: nb 64: 171.784, nb 128: 159.849, nb 256: 158.109, nb 384: 161.688, nb 512: 164.032
    {3, 1073741824, 256},  // f32, measured at n = 32768: nb 64: 1200.106, nb 128: 1107.765, nb 256: 1089.696, nb 384: 1095.953, nb 512: 1099.100
};

}  // namespace gb
