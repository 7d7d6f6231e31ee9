// The paper's own LU variant: no pivoting on a diagonally dominant A (HPL-AI
// rules, arxiv 2202.13995, section "High Performance Linpack"), with the four
// per-block operations of its "Base Implementation" (figure "lu_iteration"):
//   LU    -- factor the diagonal block,
//   top   -- A12 <- L11^-1 A12           (trsm_lower_kernel, panel.cu),
//   left  -- A21 <- A21 U11^-1           (below_solve_kernel, here),
//   inner -- A22 <- A22 - A21 A12        (the trailing-update GEMMs).
// Without pivoting no column needs a search over all rows, so the latency of
// the partial-pivot panel disappears; the price is stability, which the
// diagonal dominance of the matrix provides.
//
// Here the "LU" and "left" operations factor a whole m x w block column
// without pivoting, slab by slab: the block column's top h rows (a slab) are
// factored by one CTA in shared memory -- the LU of the slab's h x h diagonal
// block and its U rows to the right -- and then every row below the slab gets
// its L columns (X <- X U^-1 for the slab's h columns) and the update of the
// block column's remaining columns, a CTA per 64 rows.  The next slab starts
// h rows and h columns further down.  The same two kernels serve the
// diagonal-pivot check of a pivoted panel (SpecArgs in kernels.h).
#include "common.cuh"
#include "kernels.h"

namespace gb {

// Device view of SpecArgs.  Flags: [0] sticky failure, [1] kabs + 1 of a panel
// whose slab failed and [2] the rows to restore then, [3] kabs + 1 of a panel
// whose rows below a slab failed (every row to restore).
template <typename T>
struct SpecDev {
  int* flag;
  T* backup;
  int* ipiv;
  int* perm;
};

template <typename T>
__device__ __forceinline__ bool spec_ok_mult(T l) {
  return l <= T(0.5) && l >= T(-0.5);  // false for NaN
}

template <typename T>
__device__ __forceinline__ bool finite_nonzero(T v) {
  return v != T(0) && v - v == T(0);
}

// 16-byte vector of T
template <typename T>
struct V16;
template <>
struct V16<float> {
  using type = float4;
  static constexpr int n = 4;
};
template <>
struct V16<double> {
  using type = double2;
  static constexpr int n = 2;
};
template <typename T>
__device__ __forceinline__ void v16_get(const typename V16<T>::type& v, T* out);
template <>
__device__ __forceinline__ void v16_get<float>(const float4& v, float* o) {
  o[0] = v.x;
  o[1] = v.y;
  o[2] = v.z;
  o[3] = v.w;
}
template <>
__device__ __forceinline__ void v16_get<double>(const double2& v, double* o) {
  o[0] = v.x;
  o[1] = v.y;
}

template <typename T>
__device__ __forceinline__ typename V16<T>::type v16_make(const T* e);
template <>
__device__ __forceinline__ float4 v16_make<float>(const float* e) {
  return make_float4(e[0], e[1], e[2], e[3]);
}
template <>
__device__ __forceinline__ double2 v16_make<double>(const double* e) {
  return make_double2(e[0], e[1]);
}

// Rows [0, nrows) x columns [0, ncol) of G (row-major, ld) into S (row
// stride sld), and, when B is set, to B too (row stride ncol).  Each warp
// takes four rows at a time with all their loads in flight; 16-byte loads
// when G's rows are 16-byte aligned.  Rows nrows .. rows_alloc of S are
// zero-filled.
template <typename T, int NT>
__device__ __forceinline__ void load_rows(const T* G, int64_t ld, int nrows, int rows_alloc, int ncol, T* S,
                                          int sld, T* B) {
  constexpr int VN = V16<T>::n;
  using VT = typename V16<T>::type;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = NT / 32;
  const bool vec = ((reinterpret_cast<uintptr_t>(G) & 15) == 0) && ((ld * (int64_t)sizeof(T)) & 15) == 0;
  const int nvec = vec ? ncol / VN : 0;  // whole vectors per row
  for (int r0 = warp * 4; r0 < rows_alloc; r0 += NW * 4) {
    // the vector part: 4 rows x 4 vectors per lane in flight at a time
    for (int v0 = 0; v0 < nvec; v0 += 32 * 4) {
      VT buf[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int r = r0 + i, v = v0 + lane + 32 * q;
          if (r < nrows && v < nvec) buf[i][q] = reinterpret_cast<const VT*>(G + (int64_t)r * ld)[v];
        }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int r = r0 + i, v = v0 + lane + 32 * q;
          if (r < rows_alloc && v < nvec) {
            T e[VN];
            if (r < nrows) {
              v16_get<T>(buf[i][q], e);
            } else {
#pragma unroll
              for (int x = 0; x < VN; ++x) e[x] = T(0);
            }
#pragma unroll
            for (int x = 0; x < VN; ++x) {
              S[(size_t)r * sld + v * VN + x] = e[x];
              if (B && r < nrows) B[(int64_t)r * ncol + v * VN + x] = e[x];
            }
          }
        }
    }
    // the scalar rest of each row
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + i;
      if (r >= rows_alloc) break;
      for (int c = nvec * VN + lane; c < ncol; c += 32) {
        const T e = r < nrows ? G[(int64_t)r * ld + c] : T(0);
        S[(size_t)r * sld + c] = e;
        if (B && r < nrows) B[(int64_t)r * ncol + c] = e;
      }
    }
  }
}

// ============================================================ slab LU
// One CTA factors the slab D (hs rows x wt columns, row-major, ld) in shared
// memory: the LU of its hs x hs diagonal block without pivoting, blocked by 32
// columns, and U's rows right of the block (columns hs .. wt).  Per block of
// 32 columns:
//   (a)  the 32 x 32 diagonal block, by one warp, a lane per row with the
//        row's 32 columns in registers: column by column, the pivot's lane
//        writes its row (U) to shared memory, every lane below it divides by
//        the pivot (as in the definition) and subtracts its multiple of the row;
//   (b)  the rows below the block, a thread per row, by the same elimination
//        against the block's finished U, and beside them, on other warps,
//        (i') U's rows right of the block by forward substitution with the
//        block's L, a thread per column;
//   (ii) a rank-32 update of the rows below the block and the columns right
//        of it, in 32 x 32 tiles, a warp per tile (8 x 4 per thread, 16-byte
//        operand loads).  Warp 0 takes the next diagonal block's tile first
//        and factors that block at once, so that (a) runs under the other
//        warps' tiles.
// Every element gets the same products in the same order as column-by-column
// rank-1 updates of the 32-column block would give it.
// Then, for the rows below the slab, (iii) the inverses of U's 32 x 32
// diagonal blocks (a warp per block, a lane per column), written to uinv while
// the other warps write the slab back.
// What bounds it: the chain of hs dependent columns on one SM.  Column steps
// across the whole CTA cost two barriers and a round through shared memory
// each (about 900 cycles); within a warp the step is a broadcast and a
// division.  The register arrays are indexed statically in bodies of eight
// columns that a rolled loop runs four times, the registers moved down by
// eight in between: a fully unrolled block would be fetched from L2.
// A zero pivot lowers *info to its absolute column + 1 (kabs = D's first
// column) and skips its scaling.  With sp.flag set it is a stage of a pivoted
// panel's diagonal-pivot check: the first slab (first != 0) saves its rows to
// sp.backup and writes the identity pivots and an empty permutation record
// for the panel's wt columns; *info is left alone; a multiplier above 1/2, or
// a zero or non-finite pivot, records the failure (flag[1] = tag, flag[2] =
// restore_rows, then flag[0]).  It returns at once when an earlier stage or
// panel failed.
constexpr int SL_THREADS = 256;
constexpr int SL_WARPS = SL_THREADS / 32;

// Row stride of the slab in shared memory, in elements: at least the width
// and whole 32-column blocks, and VN (mod 2 VN) for VN elements per 16 bytes,
// so that the 16-byte pieces that a quarter-warp reads from eight consecutive
// rows fall in different banks.
__host__ __device__ inline int slab_wp(int hs, int wt, int tsize) {
  const int vn = 16 / tsize;
  const int w = wt > ((hs + 31) & ~31) ? wt : ((hs + 31) & ~31);
  return (w + 2 * vn - 1) / (2 * vn) * (2 * vn) + vn;
}
inline size_t slab_smem_bytes(int hs, int wt, int tsize) { return (size_t)hs * slab_wp(hs, wt, tsize) * tsize; }

// VN consecutive elements of shared memory (16-byte aligned) from / to registers
template <typename T>
__device__ __forceinline__ void s16_get(const T* p, T* out) {
  v16_get<T>(*reinterpret_cast<const typename V16<T>::type*>(p), out);
}
template <typename T>
__device__ __forceinline__ void s16_put(T* p, const T* e) {
  *reinterpret_cast<typename V16<T>::type*>(p) = v16_make<T>(e);
}

// Eliminate the 32 columns c0 .. c0 + bw of this thread's row (at `row`, the
// row's column c0; bw < 32 only for a ragged last block) against the rows of
// U of the diagonal block at Ub (row stride wp).  DIAG: the warp's lanes are
// the diagonal block's own rows, lane j publishing row j before column j's
// step; `live` lanes hold a row.
template <typename T, bool DIAG>
__device__ __forceinline__ void slab_eliminate(T* Ub, int wp, T* row, bool live, int bw, bool spec, int* info, int kcol,
                                               bool& bad) {
  constexpr int VN = V16<T>::n;
  const int lane = threadIdx.x & 31;
  T a[32];
#pragma unroll
  for (int g = 0; g < 32 / VN; ++g) {
    if (live) {
      s16_get<T>(row + g * VN, a + g * VN);
    } else {
#pragma unroll
      for (int e = 0; e < VN; ++e) a[g * VN + e] = T(0);
    }
  }
#pragma unroll 1
  for (int jb = 0; jb < 32; jb += 8) {
    if (jb >= bw) break;
    const int left = 32 - jb;  // columns jb .. 31 are in a[0 .. left)
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) {
      const int j = jb + jj;
      if (j < bw) {
        T* urow = Ub + (size_t)j * wp + jb;
        if (DIAG) {
          if (lane == j) {
#pragma unroll
            for (int g = jj / VN; g < 32 / VN; ++g)
              if (g * VN < left) s16_put<T>(urow + g * VN, a + g * VN);
          }
          __syncwarp();
        }
        T u[32];
#pragma unroll
        for (int g = jj / VN; g < 32 / VN; ++g)
          if (g * VN < left) s16_get<T>(urow + g * VN, u + g * VN);
        const T piv = u[jj];
        const bool pz = !(piv != T(0));
        if (DIAG && lane == 0) {
          if (spec) {
            if (!finite_nonzero(piv)) bad = true;
          } else if (pz) {
            atomicMin(info, kcol + j + 1);
          }
        }
        if (live && (!DIAG || lane > j)) {
          T l = a[jj];
          if (!pz) l = l / piv;
          if (spec && !spec_ok_mult(l)) bad = true;
          a[jj] = l;
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            if (g * 8 < left) {  // uniform
#pragma unroll
              for (int e = 0; e < 8; ++e)
                if (g * 8 + e > jj) a[g * 8 + e] = fma(-l, u[g * 8 + e], a[g * 8 + e]);
            }
          }
        }
      }
    }
    if (live) {
#pragma unroll
      for (int g = 0; g < 8 / VN; ++g) s16_put<T>(row + jb + g * VN, a + g * VN);
    }
#pragma unroll
    for (int i = 0; i < 24; ++i) a[i] = a[i + 8];
  }
  if (DIAG) __syncwarp();
}

// Column of U's 32 rows right of a diagonal block: x <- L^-1 x, x_t at
// x[t * wp], L (unit lower, 32 x 32) at Lb.
template <typename T>
__device__ __forceinline__ void slab_top_column(const T* Lb, int wp, T* xcol) {
  constexpr int VN = V16<T>::n;
  T x[32];
#pragma unroll
  for (int t = 0; t < 32; ++t) x[t] = xcol[(size_t)t * wp];
#pragma unroll 1
  for (int sb = 0; sb < 32; sb += 8) {
    const int left = 32 - sb;  // rows sb .. 31 are in x[0 .. left)
#pragma unroll
    for (int i = 1; i < 32; ++i) {
      if (i < left) {  // uniform
        T l[8];
#pragma unroll
        for (int g = 0; g < 8 / VN; ++g) s16_get<T>(Lb + (size_t)(sb + i) * wp + sb + g * VN, l + g * VN);
#pragma unroll
        for (int s = 0; s < 8; ++s)
          if (s < i) x[i] = fma(-l[s], x[s], x[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) xcol[(size_t)(sb + i) * wp] = x[i];
#pragma unroll
    for (int i = 0; i < 24; ++i) x[i] = x[i + 8];
  }
}

// One warp: the 32 x 32 tile of A at rows rr.., columns cc.. -= (the rows'
// columns c0 .. c0 + 31) x (rows c0 .. c0 + 31's columns).  Thread = rows
// rr + (lane >> 3) + 4 i, columns cc + 4 (lane & 7) ..: the four row groups'
// 16-byte pieces fall in different banks.
template <typename T>
__device__ __forceinline__ void slab_update_tile(T* A, int wp, int c0, int rr, int cc, int hs, int wt) {
  constexpr int VN = V16<T>::n;
  const int lane = threadIdx.x & 31;
  const int r0 = rr + (lane >> 3), cj = cc + 4 * (lane & 7);
  if (cj >= wt) return;  // (columns past wt but below its 16-byte piece's end are padding of the row)
  T acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[i][q] = T(0);
  const T* ar[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) ar[i] = A + (size_t)min(r0 + 4 * i, hs - 1) * wp + c0;
  const T* br = A + (size_t)c0 * wp + cj;
#pragma unroll 1
  for (int k = 0; k < 32; k += VN) {
    T av[8][VN];
#pragma unroll
    for (int i = 0; i < 8; ++i) s16_get<T>(ar[i] + k, av[i]);
#pragma unroll
    for (int e = 0; e < VN; ++e) {
      T bv[4];
#pragma unroll
      for (int q = 0; q < 4; q += VN) s16_get<T>(br + (size_t)(k + e) * wp + q, bv + q);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][q] = fma(av[i][e], bv[q], acc[i][q]);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = r0 + 4 * i;
    if (r < hs) {
      T* p = A + (size_t)r * wp + cj;
#pragma unroll
      for (int q = 0; q < 4; q += VN) {
        T y[VN];
        s16_get<T>(p + q, y);
#pragma unroll
        for (int e = 0; e < VN; ++e) y[e] -= acc[i][q + e];
        s16_put<T>(p + q, y);
      }
    }
  }
}

// One warp: the inverse of the upper bw x bw block Ub (row stride wp) to out
// (32 x 32, row-major; the identity outside a ragged block).  Lane = a column
// of the inverse: back substitution with the division by U's diagonal.
template <typename T>
__device__ __forceinline__ void slab_inverse(const T* Ub, int wp, int bw, T* out) {
  const int lane = threadIdx.x & 31;
  T z[32];  // row tb + i of the column at z[24 + i]
#pragma unroll
  for (int t = 0; t < 32; ++t) z[t] = t == lane ? T(1) : T(0);
#pragma unroll 1
  for (int tb = 24; tb >= 0; tb -= 8) {
#pragma unroll
    for (int jj = 7; jj >= 0; --jj) {
      const int t = tb + jj;
      if (t < bw) {  // uniform
        const T* ucol = Ub + t;  // U(q, t) at ucol[q * wp]
        const T zt = z[24 + jj] / ucol[(size_t)t * wp];
        z[24 + jj] = zt;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if (g * 8 >= 24 - tb) {  // uniform: rows tb - 24 + 8 g .. exist
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const int i = g * 8 + e;  // row q = tb - 24 + i
              if (i < 24 + jj) z[i] = z[i] - ucol[(size_t)(tb - 24 + i) * wp] * zt;
            }
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) out[(tb + i) * 32 + lane] = z[24 + i];
#pragma unroll
    for (int i = 31; i >= 8; --i) z[i] = z[i - 8];
  }
}

template <typename T>
__global__ void __launch_bounds__(SL_THREADS) slab_lu_kernel(T* D, int64_t ld, int hs, int wt, int kabs, int* info,
                                                             SpecDev<T> sp, int first, int tag, int restore_rows,
                                                             T* uinv) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int VN = V16<T>::n;
  using VT = typename V16<T>::type;
  const int wp = slab_wp(hs, wt, sizeof(T));
  T* A = reinterpret_cast<T*>(smem_raw);  // [hs][wp]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool spec = sp.flag != nullptr;
  bool bad = false;
  if (spec) {
    const int f0 = __ldcg(sp.flag), f3 = __ldcg(sp.flag + 3);
    if (f0 != 0 || f3 != 0) {
      if (tid == 0 && f0 == 0) sp.flag[0] = 1;  // a failure of the rows below an earlier slab
      return;
    }
  }
  load_rows<T, SL_THREADS>(D, ld, hs, hs, wt, A, wp, (spec && first) ? sp.backup : nullptr);
  if (spec && first) {
    for (int j = tid; j < wt; j += SL_THREADS) sp.ipiv[kabs + j] = kabs + j + 1;
    if (tid == 0) sp.perm[0] = 0;
  }
  __syncthreads();
  if (warp == 0)
    slab_eliminate<T, true>(A, wp, A + (size_t)lane * wp, lane < hs, min(32, hs), spec, info, kabs, bad);
  __syncthreads();
  for (int c0 = 0; c0 < hs; c0 += 32) {
    const int bw = min(32, hs - c0);
    const int r1 = c0 + bw;
    T* Ub = A + (size_t)c0 * wp + c0;
    // (b), (i'): rows below, then columns right of the block (a column exists
    // only beside a whole 32-column block)
    const int nr = hs - r1, nc = wt - r1;
    for (int it = tid; it < nr + nc; it += SL_THREADS) {
      if (it < nr)
        slab_eliminate<T, false>(Ub, wp, A + (size_t)(r1 + it) * wp + c0, true, bw, spec, info, kabs + c0, bad);
      else
        slab_top_column<T>(Ub, wp, A + (size_t)c0 * wp + r1 + (it - nr));
    }
    __syncthreads();
    if (nr > 0) {
      // (ii), and (a) of the next block on warp 0
      const int tc = (nc + 31) / 32, tiles = ((nr + 31) / 32) * tc;
      if (warp == 0) {
        slab_update_tile<T>(A, wp, c0, r1, r1, hs, wt);
        __syncwarp();
        slab_eliminate<T, true>(A + (size_t)r1 * wp + r1, wp, A + (size_t)min(r1 + lane, hs - 1) * wp + r1,
                                r1 + lane < hs, min(32, hs - r1), spec, info, kabs + r1, bad);
      }
      for (int t = warp == 0 ? tiles : warp; t < tiles; t += SL_WARPS - 1)
        slab_update_tile<T>(A, wp, c0, r1 + 32 * (t / tc), r1 + 32 * (t % tc), hs, wt);
      __syncthreads();
    }
  }
  // (iii) on the first warps while the others write the slab back
  const int nblk = uinv != nullptr ? (hs + 31) / 32 : 0;
  const int w0 = nblk < SL_WARPS ? nblk : 0;
  if (warp >= w0) {
    const bool vec = ((reinterpret_cast<uintptr_t>(D) & 15) == 0) && ((ld * (int64_t)sizeof(T)) & 15) == 0;
    const int nvec = vec ? wt / VN : 0;
    for (int r = warp - w0; r < hs; r += SL_WARPS - w0) {
      for (int v = lane; v < nvec; v += 32)
        reinterpret_cast<VT*>(D + (int64_t)r * ld)[v] = *reinterpret_cast<const VT*>(A + (size_t)r * wp + v * VN);
      for (int c = nvec * VN + lane; c < wt; c += 32) D[(int64_t)r * ld + c] = A[(size_t)r * wp + c];
    }
  }
  for (int b = warp; b < nblk; b += SL_WARPS)
    slab_inverse<T>(A + (size_t)(32 * b) * wp + 32 * b, wp, min(32, hs - 32 * b), uinv + (size_t)b * 1024);
  if (spec && __syncthreads_or(bad) && tid == 0) {
    sp.flag[1] = tag;
    sp.flag[2] = restore_rows;
    __threadfence();
    sp.flag[0] = 1;
  }
}

// ============================================================ rows below a slab
// X (m x wt, row-major, ld): the ws columns of a slab's rows below it are
// solved against the slab's upper ws x ws block U (X <- X U^-1, the paper's
// "left" block update) and the other wt - ws columns updated with U's rows
// right of the block (U is ws x wt at U, row-major, ld).  CTA = RB rows of X
// in shared memory; by 32-column blocks of the ws:
//   1. U's 32 rows of the block staged in shared memory (cp.async);
//   2. the diagonal block: X_b <- X_b U_bb^-1, a small product with the
//      inverse of U's 32 x 32 diagonal block, which the slab kernel wrote to
//      uinv (32 x 32 per block, row-major);
//   3. the columns to the right: a rank-32 update, each thread a register
//      tile of RB/16 rows x 4 columns per 64-column chunk, its rows' values
//      of the block read from a transposed copy (one 16-byte load per k).
// With sp.flag set it is a stage of the diagonal-pivot check: for the first
// slab (first != 0) the rows are saved to sp.backup first and the stage runs
// unless flag[0] is set; a later stage returns on flag[0] or flag[3].  A
// multiplier above 1/2 in magnitude (or not finite) records flag[3] = tag.
constexpr int LS_THREADS = 256;

template <typename T, int RB>
__global__ void __launch_bounds__(LS_THREADS) below_solve_kernel(const T* __restrict__ U, const T* __restrict__ uinv,
                                                                 T* X, int64_t ld, int m, int ws, int wt,
                                                                 SpecDev<T> sp, int first, int tag) {
  static_assert(RB % 16 == 0 && RB <= LS_THREADS, "RB rows: 16 row groups, one thread per row");
  constexpr int RT = RB / 16;  // rows per thread in the update
  constexpr int VN = V16<T>::n;
  using VT = typename V16<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int wx = wt | 1;          // odd row stride: a row per thread is free of bank conflicts
  const int wu = (wt + 3) & ~3;   // U stage row stride: 16-byte rows
  T* Us = reinterpret_cast<T*>(smem_raw);  // [32][wu]: rows c0 .. c0 + 31 of U, columns c0 .. wt
  T* Ui = Us + 32 * wu;                    // [32][32]: the inverse of U's current 32 x 32 diagonal block
  T* Xs = Ui + 32 * 32;                    // [RB][wx]
  T* XT = Xs + RB * wx;                    // [32][RB]: the solved block, transposed (16-byte aligned)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = blockIdx.x * RB;
  const int rows = min(RB, m - r0);
  const bool spec = sp.flag != nullptr;
  if (spec) {
    const bool stop = first ? __ldcg(sp.flag) != 0 : (__ldcg(sp.flag) != 0 || __ldcg(sp.flag + 3) != 0);
    if (stop) return;
  }
  bool bad = false;
  const bool uvec = ((reinterpret_cast<uintptr_t>(U) & 15) == 0) && ((ld * (int64_t)sizeof(T)) & 15) == 0;
  load_rows<T, LS_THREADS>(X + (int64_t)r0 * ld, ld, rows, RB, wt, Xs, wx,
                           (spec && first) ? sp.backup + (int64_t)r0 * wt : nullptr);
  for (int c0 = 0; c0 < ws; c0 += 32) {
    const int bw = min(32, ws - c0);
    __syncthreads();  // the previous block's update is done with Us
    // U's rows c0 .. c0 + bw, columns c0 .. wt: asynchronous copies, all in flight together
    {
      const int nv = uvec ? (wt - c0) / VN : 0;  // c0 is a multiple of 32: 16-byte aligned when U's rows are
      for (int e = tid; e < bw * nv; e += LS_THREADS) {
        const int k = e / nv, v = e % nv;
        cp_async<16>(&Us[k * wu + c0 + v * VN], &U[(int64_t)(c0 + k) * ld + c0 + v * VN]);
      }
      const int done = c0 + nv * VN, rest = wt - done;
      for (int e = tid; e < bw * rest; e += LS_THREADS) {
        const int k = e / rest, c = done + e % rest;
        cp_async<sizeof(T)>(&Us[k * wu + c], &U[(int64_t)(c0 + k) * ld + c]);
      }
      const T* ub = uinv + (size_t)(c0 / 32) * 1024;
      for (int e = tid; e < 1024 / VN; e += LS_THREADS) cp_async<16>(&Ui[e * VN], &ub[e * VN]);
      cp_async_wait_all();
    }
    __syncthreads();
    // the diagonal block: X_b <- X_b Ui, a small product over the whole CTA
    // (rows x quads of columns; results held until every thread has read)
    {
      T res[(RB * 8 + LS_THREADS - 1) / LS_THREADS][4];
#pragma unroll
      for (int it = 0; it < (RB * 8 + LS_THREADS - 1) / LS_THREADS; ++it) {
        const int e = tid + it * LS_THREADS;
        const int r = e >> 3, cq = (e & 7) * 4;
#pragma unroll
        for (int q = 0; q < 4; ++q) res[it][q] = T(0);
        if (e < RB * 8) {
#pragma unroll 8
          for (int k = 0; k < bw; ++k) {
            const T xk = Xs[r * wx + c0 + k];
            T uv[4];
            v16_get<T>(*reinterpret_cast<const VT*>(&Ui[k * 32 + cq]), uv);
            if (VN == 2) v16_get<T>(*reinterpret_cast<const VT*>(&Ui[k * 32 + cq + 2]), uv + 2);
#pragma unroll
            for (int q = 0; q < 4; ++q) res[it][q] = fma(xk, uv[q], res[it][q]);
          }
        }
      }
      __syncthreads();
#pragma unroll
      for (int it = 0; it < (RB * 8 + LS_THREADS - 1) / LS_THREADS; ++it) {
        const int e = tid + it * LS_THREADS;
        const int r = e >> 3, cq = (e & 7) * 4;
        if (e < RB * 8) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (cq + q < bw) {
              Xs[r * wx + c0 + cq + q] = res[it][q];
              if (spec && r < rows && !spec_ok_mult(res[it][q])) bad = true;
            }
          }
        }
      }
    }
    __syncthreads();
    for (int e = tid; e < 32 * RB; e += LS_THREADS) {
      const int k = e / RB, r = e % RB;
      XT[k * RB + r] = k < bw ? Xs[r * wx + c0 + k] : T(0);
    }
    __syncthreads();
    const int c1 = c0 + bw;  // columns [c1, wt) remain
    const int rg = tid >> 4, cg = tid & 15;
    for (int cc = c1 + 4 * cg; cc < wt; cc += 64) {
      T acc[RT][4];
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][q] = T(0);
#pragma unroll 4
      for (int k = 0; k < bw; ++k) {
        // columns past wt are never stored; c1 and cc are multiples of 4 (a
        // remaining column exists only after a full 32-column block), so the
        // 16-byte loads stay inside the stage's 16-byte rows
        T ub[4], xa[RT];
        const T* up = &Us[k * wu + cc];
        v16_get<T>(*reinterpret_cast<const VT*>(up), ub);
        if (VN == 2) v16_get<T>(*reinterpret_cast<const VT*>(up + 2), ub + 2);
        if constexpr (RT % VN == 0) {
#pragma unroll
          for (int i = 0; i < RT; i += VN) v16_get<T>(*reinterpret_cast<const VT*>(&XT[k * RB + RT * rg + i]), xa + i);
        } else {
#pragma unroll
          for (int i = 0; i < RT; ++i) xa[i] = XT[k * RB + RT * rg + i];
        }
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[i][q] = fma(xa[i], ub[q], acc[i][q]);
      }
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (cc + q < wt) Xs[(RT * rg + i) * wx + cc + q] -= acc[i][q];
    }
  }
  __syncthreads();
  for (int r = warp; r < rows; r += LS_THREADS / 32)
    for (int c = lane; c < wt; c += 32) X[(int64_t)(r0 + r) * ld + c] = Xs[r * wx + c];
  if (spec && __syncthreads_or(bad) && tid == 0) sp.flag[3] = tag;
}

// ============================================================ launchers
template <typename T>
static SpecDev<T> spec_dev(const SpecArgs& a, int64_t backup_offset) {
  SpecDev<T> d;
  d.flag = a.flag;
  d.backup = a.backup ? reinterpret_cast<T*>(a.backup) + backup_offset : nullptr;
  d.ipiv = a.ipiv;
  d.perm = a.perm;
  return d;
}

static int device_smem_optin() {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return optin;
}

// Slab height: the largest multiple of 32, at most 128, whose slab fits in
// 168 KB of shared memory.
static int slab_rows(int w, int tsize) {
  int h = 128;
  while (h > 32 && slab_smem_bytes(h, w, tsize) > 168 * 1024) h -= 32;
  return h;
}

static size_t ls_smem(int rb, int wt, int tsize) {
  const size_t wu = (size_t)((wt + 3) & ~3);
  return (32 * wu + 32 * 32 + (size_t)rb * (wt | 1) + 32 * (size_t)rb) * tsize;
}

template <typename T, int RB>
static cudaError_t launch_ls(const T* U, const T* uinv, T* X, int64_t ld, int m, int ws, int wt,
                             const SpecDev<T>& sp, int first, int tag, cudaStream_t st) {
  auto kern = below_solve_kernel<T, RB>;
  cudaError_t e = allow_max_smem((const void*)kern);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)cdiv(m, RB), LS_THREADS, ls_smem(RB, wt, sizeof(T)), st>>>(U, uinv, X, ld, m, ws, wt, sp, first,
                                                                               tag);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_below(const T* U, const T* uinv, T* X, int64_t ld, int m, int ws, int wt,
                                const SpecDev<T>& sp, int first, int tag, cudaStream_t st) {
  const int optin = device_smem_optin();
  if (ls_smem(64, wt, sizeof(T)) <= (size_t)optin)
    return launch_ls<T, 64>(U, uinv, X, ld, m, ws, wt, sp, first, tag, st);
  if (ls_smem(32, wt, sizeof(T)) <= (size_t)optin)
    return launch_ls<T, 32>(U, uinv, X, ld, m, ws, wt, sp, first, tag, st);
  if (ls_smem(16, wt, sizeof(T)) <= (size_t)optin)
    return launch_ls<T, 16>(U, uinv, X, ld, m, ws, wt, sp, first, tag, st);
  return cudaErrorInvalidValue;
}

// One slab: a CTA with the slab in shared memory.
template <typename T>
static cudaError_t launch_slab(T* D, int64_t ld, int hs, int wt, int kabs, int* info, const SpecDev<T>& sp,
                               int first, int tag, int restore, T* uinv, cudaStream_t st) {
  auto kern = slab_lu_kernel<T>;
  cudaError_t e = allow_max_smem((const void*)kern);
  if (e != cudaSuccess) return e;
  kern<<<1, SL_THREADS, slab_smem_bytes(hs, wt, sizeof(T)), st>>>(D, ld, hs, wt, kabs, info, sp, first, tag, restore,
                                                                   uinv);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_block_column(T* P, int64_t ld, int m, int w, int kabs, int* info, T* uinv, cudaStream_t st,
                                const SpecArgs& spec) {
  if (w <= 0) return cudaSuccess;
  if (m < w) return cudaErrorInvalidValue;
  const int h = slab_rows(w, sizeof(T));
  cudaError_t e = cudaSuccess;
  const int tag = kabs + 1;
  for (int s0 = 0; s0 < w; s0 += h) {
    const int hs = (w - s0) < h ? (w - s0) : h;
    const int wt = w - s0;
    const int first = s0 == 0;
    T* D = P + (int64_t)s0 * ld + s0;
    // a failed check of the first slab changed only its rows; any later
    // failure, every row of the block column
    const int restore = first ? hs : m;
    const int below = m - s0 - hs;
    T* ui = uinv + (size_t)(s0 / 32) * 1024;  // the slab's diagonal blocks' inverses (for the rows below)
    if ((e = launch_slab<T>(D, ld, hs, wt, kabs + s0, info, spec_dev<T>(spec, 0), first, tag, restore,
                            below > 0 ? ui : nullptr, st)) != cudaSuccess)
      return e;
    if (below > 0) {
      // the first slab's rows below it follow its rows in the backup (row stride w)
      e = launch_below<T>(D, ui, D + (int64_t)hs * ld, ld, below, hs, wt, spec_dev<T>(spec, (int64_t)hs * w), first,
                          tag, st);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

int block_column_launches(int m, int w, int tsize) {
  if (w <= 0) return 0;
  const int h = slab_rows(w, tsize);
  int n = 0;
  for (int s0 = 0; s0 < w; s0 += h) {
    const int hs = (w - s0) < h ? (w - s0) : h;
    n += (m - s0 - hs) > 0 ? 2 : 1;
  }
  return n;
}

template cudaError_t launch_block_column<double>(double*, int64_t, int, int, int, int*, double*, cudaStream_t,
                                                 const SpecArgs&);
template cudaError_t launch_block_column<float>(float*, int64_t, int, int, int, int*, float*, cudaStream_t,
                                                const SpecArgs&);

}  // namespace gb
