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
    {0, 800, 64},  // f64, measured at n = 600: nb 32: 1.680, nb 64: 1.585, nb 96: 1.600, nb 128: 1.640, nb 192: 1.852, nb 256: 2.035
    {0, 1280, 64},  // f64, measured at n = 1023: nb 32: 3.286, nb 64: 3.083, nb 96: 3.131, nb 128: 3.314, nb 192: 3.611, nb 256: 3.920
    {0, 3072, 128},  // f64, measured at n = 2048: nb 32: 11.199, nb 64: 7.896, nb 96: 7.569, nb 128: 7.360, nb 192: 7.743, nb 256: 8.409
    {0, 4608, 128},  // f64, measured at n = 4096: nb 32: 53.185, nb 64: 23.485, nb 96: 20.599, nb 128: 19.022, nb 192: 18.948, nb 256: 19.644
    {0, 7168, 192},  // f64, measured at n = 6000: nb 32: 145.067, nb 64: 50.690, nb 96: 41.958, nb 128: 36.996, nb 192: 34.807, nb 256: 35.107
    {0, 12288, 256},  // f64, measured at n = 8192: nb 32: 340.921, nb 64: 101.347, nb 96: 79.956, nb 128: 68.142, nb 192: 60.611, nb 256: 59.217
    {0, 24576, 256},  // f64, measured at n = 16384: nb 32: 2521.305, nb 64: 608.801, nb 96: 447.020, nb 128: 361.227, nb 192: 289.931, nb 256: 260.948
    {0, 1073741824, 256},  // f64, measured at n = 32768: not measured: n = 32768 keeps the smaller size's choice
    {1, 1280, 128},  // f64_split, measured at n = 1024: nb 64: 4.663, nb 128: 4.065, nb 192: 4.094, nb 256: 4.206
    {1, 3072, 128},  // f64_split, measured at n = 2048: nb 64: 10.488, nb 128: 8.692, nb 192: 8.566, nb 256: 8.808
    {1, 4608, 256},  // f64_split, measured at n = 4096: nb 64: 27.908, nb 128: 21.090, nb 192: 19.890, nb 256: 19.625
    {1, 7168, 256},  // f64_split, measured at n = 7001: nb 64: 76.885, nb 128: 51.887, nb 192: 45.207, nb 256: 43.258
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
