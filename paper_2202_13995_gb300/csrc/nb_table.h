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
    {0, 1536, 64},  // f64, measured at n = 1023: nb 64: 4.59, nb 128: 4.70, nb 192: 5.48, nb 256: 6.43
    {0, 3072, 64},  // f64, measured at n = 2048: nb 64: 10.46, nb 128: 10.86, nb 192: 13.50, nb 256: 16.22 (3000: 17.9, 19.1, 22.6, 25.4)
    {0, 6144, 128},  // f64, measured at n = 6000: nb 64: 61.05, nb 128: 55.45, nb 192: 58.05, nb 256: 62.07 (4096: 29.4, 30.1, 34.1, 37.4)
    {0, 12288, 192},  // f64, measured at n = 8192: nb 64: 118.4, nb 128: 94.89, nb 192: 93.46, nb 256: 96.34
    {0, 24576, 256},  // f64, measured at n = 16384: nb 64: 647, nb 128: 412, nb 192: 349, nb 256: 326
    {0, 1073741824, 256},  // f64, measured at n = 32768: not measured: n = 32768 keeps the smaller size's choice
    {1, 1536, 128},  // f64_split, measured at n = 1024: nb 64: 8.105, nb 128: 7.824, nb 192: 8.141, nb 256: 8.463
    {1, 3072, 128},  // f64_split, measured at n = 2048: nb 64: 17.218, nb 128: 16.488, nb 192: 16.861, nb 256: 17.595
    {1, 6144, 128},  // f64_split, measured at n = 4096: nb 64: 40.321, nb 128: 36.240, nb 192: 36.390, nb 256: 37.338
    {1, 12288, 256},  // f64_split, measured at n = 8192: nb 64: 126.705, nb 128: 97.123, nb 192: 89.998, nb 256: 89.571
    {1, 24576, 256},  // f64_split, measured at n = 16384: nb 64: 612.232, nb 128: 384.506, nb 192: 315.130, nb 256: 290.955
    {1, 1073741824, 256},  // f64_split, measured at n = 32768: nb 64: 4066.466, nb 128: 2244.717, nb 192: 1653.813, nb 256: 1410.500
    {2, 1536, 128},  // mixed, measured at n = 1024: nb 64: 2.250, nb 128: 1.878, nb 256: 1.907, nb 384: 2.120, nb 512: 2.296
    {2, 3072, 128},  // mixed, measured at n = 2048: nb 64: 4.353, nb 128: 3.611, nb 256: 3.740, nb 384: 4.251, nb 512: 4.577
    {2, 6144, 128},  // mixed, measured at n = 4096: nb 64: 8.707, nb 128: 7.251, nb 256: 7.540, nb 384: 8.548, nb 512: 9.339
    {2, 12288, 128},  // mixed, measured at n = 8192: nb 64: 18.442, nb 128: 14.909, nb 256: 15.422, nb 384: 17.611, nb 512: 19.232
    {2, 24576, 256},  // mixed, measured at n = 16384: nb 64: 57.322, nb 128: 38.633, nb 256: 37.393, nb 384: 41.425, nb 512: 45.651
    {2, 1073741824, 256},  // mixed, measured at n = 32768: nb 64: 299.866, nb 128: 171.840, nb 256: 127.095, nb 384: 127.630, nb 512: 136.121
    {3, 1536, 128},  // f32, measured at n = 1024: nb 64: 2.038, nb 128: 1.813, nb 256: 1.914, nb 384: 2.110, nb 512: 2.303
    {3, 3072, 128},  // f32, measured at n = 2048: nb 64: 4.132, nb 128: 3.671, nb 256: 3.885, nb 384: 4.408, nb 512: 4.725
    {3, 6144, 128},  // f32, measured at n = 4096: nb 64: 9.820, nb 128: 8.795, nb 256: 9.141, nb 384: 10.152, nb 512: 10.877
    {3, 12288, 128},  // f32, measured at n = 8192: nb 64: 33.212, nb 128: 29.993, nb 256: 30.284, nb 384: 32.196, nb 512: 33.427
    {3, 24576, 256},  // f32, measured at n = 16384: nb 64: 171.784, nb 128: 159.849, nb 256: 158.109, nb 384: 161.688, nb 512: 164.032
    {3, 1073741824, 256},  // f32, measured at n = 32768: nb 64: 1200.106, nb 128: 1107.765, nb 256: 1089.696, nb 384: 1095.953, nb 512: 1099.100
};

}  // namespace gb
