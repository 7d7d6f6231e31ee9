// Block width nb of lu_factor(nb = 0), by factorization kind and size:
// chosen from sweeps of whole solves (factor + solve or refinement) on the
// benchmarks' seeded matrices, by
//   python -m paper_2202_13995_gb300.tune
// on NVIDIA GB300: the fastest width at the size, or a narrower one within 3 percent
// of it that the sizes beside it prefer (chosen by hand; the sweep names the fastest).
// Times in ms, best of five after a warm-up, all rows of one run.
#pragma once

namespace gb {

// kind: 0 FP64 (certified split update), 1 FP64 (split tensor-core update),
// 2 BF16 / FP16 mixed, 3 FP32.  The first entry of the kind whose nmax
// is at least n applies.
struct NbEntry {
  int kind, nmax, nb;
};

constexpr NbEntry kNbTable[] = {
    {0, 800, 64},  // f64, measured at n = 600: nb 32: 1.632, nb 64: 1.550, nb 96: 1.554, nb 128: 1.617, nb 192: 1.816, nb 256: 2.017
    {0, 1280, 64},  // f64, measured at n = 1024: nb 32: 3.240, nb 64: 3.058, nb 96: 3.071, nb 128: 3.096, nb 192: 3.360, nb 256: 3.715
    {0, 3072, 128},  // f64, measured at n = 2048: nb 32: 10.989, nb 64: 7.677, nb 96: 7.353, nb 128: 7.174, nb 192: 7.466, nb 256: 8.160
    {0, 4608, 128},  // f64, measured at n = 4096: nb 32: 52.866, nb 64: 22.980, nb 96: 20.144, nb 128: 18.520, nb 192: 18.478, nb 256: 19.094
    {0, 7168, 192},  // f64, measured at n = 5800: nb 32: 132.476, nb 64: 46.292, nb 96: 38.253, nb 128: 34.382, nb 192: 32.050, nb 256: 32.026
    {0, 12288, 256},  // f64, measured at n = 8192: nb 32: 339.936, nb 64: 99.328, nb 96: 78.020, nb 128: 66.484, nb 192: 58.849, nb 256: 56.148
    {0, 24576, 256},  // f64, measured at n = 16384: nb 32: 2520.064, nb 64: 597.495, nb 96: 433.155, nb 128: 345.725, nb 192: 273.029, nb 256: 235.283
    {0, 1073741824, 256},  // f64, measured at n = 32768: not measured: n = 32768 keeps the smaller size's choice
    {1, 800, 128},  // f64_split, measured at n = 600: nb 64: 2.682, nb 128: 2.132, nb 192: 2.194, nb 256: 2.268
    {1, 1280, 128},  // f64_split, measured at n = 1024: nb 64: 4.605, nb 128: 3.834, nb 192: 3.870, nb 256: 3.974
    {1, 3072, 128},  // f64_split, measured at n = 2048: nb 64: 10.293, nb 128: 8.450, nb 192: 8.212, nb 256: 8.491
    {1, 4608, 256},  // f64_split, measured at n = 4096: nb 64: 27.399, nb 128: 20.475, nb 192: 19.265, nb 256: 19.022
    {1, 7168, 256},  // f64_split, measured at n = 5800: nb 64: 51.732, nb 128: 36.440, nb 192: 32.254, nb 256: 31.404
    {1, 12288, 256},  // f64_split, measured at n = 8192: nb 64: 105.555, nb 128: 67.888, nb 192: 57.250, nb 256: 53.658
    {1, 24576, 256},  // f64_split, measured at n = 16384: nb 64: 596.455, nb 128: 336.324, nb 192: 257.725, nb 256: 221.104
    {1, 1073741824, 256},  // f64_split, measured at n = 32768: nb 64: 4272.015, nb 128: 2274.564, nb 192: 1668.054, nb 256: 1374.150
    {2, 800, 128},  // mixed, measured at n = 600: nb 64: 0.851, nb 128: 0.691, nb 192: 0.727, nb 256: 0.705, nb 384: 0.699, nb 512: 0.721
    {2, 1280, 256},  // mixed, measured at n = 1024: nb 64: 1.139, nb 128: 0.929, nb 192: 0.928, nb 256: 0.901, nb 384: 0.919, nb 512: 0.938
    {2, 3072, 256},  // mixed, measured at n = 2048: nb 64: 2.155, nb 128: 1.714, nb 192: 1.685, nb 256: 1.674, nb 384: 1.724, nb 512: 1.792
    {2, 4608, 256},  // mixed, measured at n = 4096: nb 64: 4.598, nb 128: 3.524, nb 192: 3.497, nb 256: 3.446, nb 384: 3.570, nb 512: 3.826
    {2, 7168, 256},  // mixed, measured at n = 5800: nb 64: 7.338, nb 128: 5.542, nb 192: 5.381, nb 256: 5.234, nb 384: 5.468, nb 512: 5.928
    {2, 12288, 256},  // mixed, measured at n = 8192: nb 64: 12.735, nb 128: 8.908, nb 192: 8.436, nb 256: 7.719, nb 384: 8.518, nb 512: 9.224
    {2, 24576, 256},  // mixed, measured at n = 16384: nb 64: 54.130, nb 128: 32.269, nb 192: 26.282, nb 256: 22.640, nb 384: 24.285, nb 512: 26.973
    {2, 1073741824, 256},  // mixed, measured at n = 32768: nb 64: 319.196, nb 128: 174.478, nb 192: 131.550, nb 256: 103.712, nb 384: 102.440, nb 512: 100.741
    {3, 800, 128},  // f32, measured at n = 600: nb 64: 0.744, nb 128: 0.647, nb 192: 0.691, nb 256: 0.685, nb 384: 0.661, nb 512: 0.756
    {3, 1280, 128},  // f32, measured at n = 1024: nb 64: 1.169, nb 128: 0.998, nb 192: 1.037, nb 256: 1.000, nb 384: 1.036, nb 512: 1.061
    {3, 3072, 128},  // f32, measured at n = 2048: nb 64: 2.342, nb 128: 2.011, nb 192: 2.037, nb 256: 2.035, nb 384: 2.185, nb 512: 2.216
    {3, 4608, 128},  // f32, measured at n = 4096: nb 64: 6.292, nb 128: 5.519, nb 192: 5.589, nb 256: 5.547, nb 384: 5.757, nb 512: 5.986
    {3, 7168, 128},  // f32, measured at n = 5800: nb 64: 12.258, nb 128: 11.036, nb 192: 10.938, nb 256: 10.945, nb 384: 11.282, nb 512: 11.667
    {3, 12288, 128},  // f32, measured at n = 8192: nb 64: 26.306, nb 128: 23.525, nb 192: 23.531, nb 256: 23.356, nb 384: 23.806, nb 512: 24.411
    {3, 24576, 256},  // f32, measured at n = 16384: nb 64: 158.769, nb 128: 147.073, nb 192: 145.933, nb 256: 144.583, nb 384: 145.465, nb 512: 146.836
    {3, 1073741824, 256},  // f32, measured at n = 32768: nb 64: 1177.684, nb 128: 1082.593, nb 192: 1071.538, nb 256: 1063.387, nb 384: 1064.212, nb 512: 1065.735
};

}  // namespace gb
