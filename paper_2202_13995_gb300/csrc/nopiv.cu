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
// block column's remaining columns, a CTA per 16 to 64 rows.  The next slab starts
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
//   (a)  the 32 x 32 diagonal block, by one warp, a lane per row, in
//        sub-blocks of eight columns held in registers: per column the pivot
//        row comes by shuffles, every lane below divides by the pivot (as in
//        the definition) and subtracts its multiple of the row; then the
//        sub-block's rows of U to its right (a lane per column) and a rank-8
//        update of the rows below (a lane per row);
//   (b)  the rows below the block, two or four lanes per row, by the same
//        elimination against the block's finished U, and beside them, on other warps,
//        (i') U's rows right of the block by forward substitution with the
//        block's L, a thread per column, both by sub-blocks of eight;
//   (ii) a rank-32 update of the rows below the block and the columns right
//        of it, in 32 x 32 tiles, a warp per tile (8 x 4 per thread, 16-byte
//        operand loads).  Warps 0 to 3 share the next diagonal block's tile
//        first and warp 0 factors that block at once, so that (a) runs under
//        the other warps' tiles.
// Every element gets the same products in the same order as column-by-column
// rank-1 updates of the 32-column block would give it.
// Then, for the rows below the slab, (iii) the inverses of U's 32 x 32
// diagonal blocks (a warp per block, a lane per column), written to uinv while
// the other warps write the slab back.
// What bounds it: the chain of hs dependent columns on one SM (clock stamps,
// 128 x 256 FP32 slab: 240 cycles a column in (a), 5000 to 7600 per block in
// (b) and (i'), 9000 for the inverses and the write-back).  Alone on the GPU a
// 128 x 256 slab takes 47 us and a 128 x 128 one 41 us; with each column step
// across the whole CTA, two barriers and a round through shared memory a
// column, they took 112 and 87 us.
// The loops over sub-blocks stay rolled and their bodies short and free of
// branches: a 32-column elimination with every column in registers measured
// 440 cycles a column, most of them at the ends of its many short branches.
// A zero pivot lowers *info to its absolute column + 1 (kabs = D's first
// column) and skips its scaling.  With sp.flag set it is a stage of a pivoted
// panel's diagonal-pivot check: the first slab (first != 0) saves its rows to
// sp.backup and writes the identity pivots and an empty permutation record
// for the panel's wt columns; *info is left alone; a multiplier above 1/2, or
// a zero or non-finite pivot, records the failure (flag[1] = tag, flag[2] =
// restore_rows, then flag[0]).  It returns at once when an earlier stage or
// panel failed.
constexpr int SL_THREADS = 512;
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
// shared memory of one slab: its rows, and 32 x 32 scratch per diagonal block for its U's inverse
inline size_t slab_smem_bytes(int hs, int wt, int tsize) {
  return ((size_t)hs * slab_wp(hs, wt, tsize) + (size_t)((hs + 31) / 32) * 1024) * tsize;
}

// VN consecutive elements of shared memory (16-byte aligned) from / to registers
template <typename T>
__device__ __forceinline__ void s16_get(const T* p, T* out) {
  v16_get<T>(*reinterpret_cast<const typename V16<T>::type*>(p), out);
}
template <typename T>
__device__ __forceinline__ void s16_put(T* p, const T* e) {
  *reinterpret_cast<typename V16<T>::type*>(p) = v16_make<T>(e);
}

// Eight columns of a row, y (registers) -= a x (eight rows of U at u, row stride wp)
template <typename T>
__device__ __forceinline__ void slab_rank8(T* y, const T (&a)[8], const T* u, int wp) {
  constexpr int VN = V16<T>::n;
  T yv[8];
#pragma unroll
  for (int g = 0; g < 8; g += VN) s16_get<T>(y + g, yv + g);
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    T uv[8];
#pragma unroll
    for (int g = 0; g < 8; g += VN) s16_get<T>(u + (size_t)t * wp + g, uv + g);
#pragma unroll
    for (int e = 0; e < 8; ++e) yv[e] = fma(-a[t], uv[e], yv[e]);
  }
#pragma unroll
  for (int g = 0; g < 8; g += VN) s16_put<T>(y + g, yv + g);
}

// One column's eight entries x (row stride wp) <- their part of L^-1 x for the
// 8 x 8 unit-lower block at L; xv keeps them
template <typename T>
__device__ __forceinline__ void slab_tri8(T* x, const T* L, int wp, T (&xv)[8]) {
  constexpr int VN = V16<T>::n;
#pragma unroll
  for (int t = 0; t < 8; ++t) xv[t] = x[(size_t)t * wp];
#pragma unroll
  for (int t = 1; t < 8; ++t) {
    T l[8];
#pragma unroll
    for (int g = 0; g < t; g += VN) s16_get<T>(L + (size_t)t * wp + g, l + g);
#pragma unroll
    for (int q = 0; q < t; ++q) xv[t] = fma(-l[q], xv[q], xv[t]);
  }
#pragma unroll
  for (int t = 1; t < 8; ++t) x[(size_t)t * wp] = xv[t];
}

// (a) One warp: LU of the bw x bw diagonal block at Ub (row stride wp; bw < 32
// only for a ragged last block), lane = row, by sub-blocks of eight columns;
// the reciprocals of its pivots to rinv.
template <typename T>
__device__ __forceinline__ void slab_diag(T* Ub, int wp, int bw, bool spec, int* info, int kcol, T* rinv, bool& bad) {
  constexpr int VN = V16<T>::n;
  const int lane = threadIdx.x & 31;
  const bool live = lane < bw;
  T* row = Ub + (size_t)lane * wp;
#pragma unroll 1
  for (int jb = 0; jb < bw; jb += 8) {
    T a[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) a[e] = T(0);
    if (live) {
#pragma unroll
      for (int g = 0; g < 8; g += VN) s16_get<T>(row + jb + g, a + g);
    }
    // lanes at or above the pivot (and lanes without a row) take part with the
    // multiplier's uses masked: no branch inside a column step
    const int below = live ? lane - jb : -1;  // columns jb + jj < lane are this row's
    const int jn = bw - jb;
    bool big = false;
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) {
      T u[8];
#pragma unroll
      for (int e = jj; e < 8; ++e) u[e] = __shfl_sync(0xffffffffu, a[e], jb + jj);
      const T l = a[jj] / (u[jj] != T(0) ? u[jj] : T(1));
      const bool upd = below > jj && jj < jn;
      big |= upd && !spec_ok_mult(l);
#pragma unroll
      for (int e = jj + 1; e < 8; ++e) a[e] = upd ? fma(-l, u[e], a[e]) : a[e];
      a[jj] = upd ? l : a[jj];
    }
    if (spec && big) bad = true;
    if (below >= 0 && below < 8) {  // this lane's row holds a pivot of the sub-block
      T piv = a[0];
#pragma unroll
      for (int e = 1; e < 8; ++e) piv = below == e ? a[e] : piv;
      rinv[lane] = recip_rn(piv);
      if (spec) {
        if (!finite_nonzero(piv)) bad = true;
      } else if (!(piv != T(0))) {
        atomicMin(info, kcol + lane + 1);
      }
    }
    if (live) {
#pragma unroll
      for (int g = 0; g < 8; g += VN) s16_put<T>(row + jb + g, a + g);
    }
    __syncwarp();
    if (jb + 8 < bw) {
      // the sub-block's rows of U right of it (lane = column), then the rows below it
      if (jb + 8 + lane < 32) {
        T x[8];
        slab_tri8<T>(Ub + (size_t)jb * wp + jb + 8 + lane, Ub + (size_t)jb * wp + jb, wp, x);
      }
      __syncwarp();
      if (live && lane >= jb + 8) {
#pragma unroll 1
        for (int cb = jb + 8; cb < 32; cb += 8) slab_rank8<T>(row + cb, a, Ub + (size_t)jb * wp + cb, wp);
      }
      __syncwarp();
    }
  }
}

// (b) Two neighbouring lanes per row: the 32 columns of a row below the
// diagonal block at Ub eliminated against its U (its pivots' reciprocals at
// rinv).  Each lane divides the sub-block's eight columns itself; the 8-column
// chunks right of them are dealt to the two lanes.
template <typename T>
__device__ __forceinline__ void slab_left_row(const T* Ub, int wp, const T* rinv, T* row, bool live, int part, bool spec,
                                              bool& bad) {
  constexpr int VN = V16<T>::n;
#pragma unroll 1
  for (int jb = 0; jb < 32; jb += 8) {
    const T* ub = Ub + (size_t)jb * wp + jb;
    T a[8];
    if (live) {
#pragma unroll
      for (int g = 0; g < 8; g += VN) s16_get<T>(row + jb + g, a + g);
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        T u[8];
#pragma unroll
        for (int g = jj / VN * VN; g < 8; g += VN) s16_get<T>(ub + (size_t)jj * wp + g, u + g);
        const T l = quot_rn(a[jj], u[jj], rinv[jb + jj]);
        if (spec && !spec_ok_mult(l)) bad = true;
        a[jj] = l;
#pragma unroll
        for (int e = jj + 1; e < 8; ++e) a[e] = fma(-l, u[e], a[e]);
      }
    }
    __syncwarp();  // every lane of the row has read the sub-block
    if (live) {
      if (part == 0) {
#pragma unroll
        for (int g = 0; g < 8; g += VN) s16_put<T>(row + jb + g, a + g);
      }
#pragma unroll 1
      for (int cb = jb + 8 + 8 * part; cb < 32; cb += 16) slab_rank8<T>(row + cb, a, ub + (cb - jb), wp);
    }
    __syncwarp();
  }
}

// (i') One thread: a column of U's 32 rows right of the diagonal block,
// x <- L^-1 x with x_t at x[t * wp] and L at Lb.
template <typename T>
__device__ __forceinline__ void slab_top_column(const T* Lb, int wp, T* x) {
  constexpr int VN = V16<T>::n;
#pragma unroll 1
  for (int sb = 0; sb < 32; sb += 8) {
    T xv[8];
    slab_tri8<T>(x + (size_t)sb * wp, Lb + (size_t)sb * wp + sb, wp, xv);
#pragma unroll 1
    for (int rb = sb + 8; rb < 32; rb += 8) {
      T y[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) y[t] = x[(size_t)(rb + t) * wp];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        T l[8];
#pragma unroll
        for (int g = 0; g < 8; g += VN) s16_get<T>(Lb + (size_t)(rb + t) * wp + sb + g, l + g);
#pragma unroll
        for (int q = 0; q < 8; ++q) y[t] = fma(-l[q], xv[q], y[t]);
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) x[(size_t)(rb + t) * wp] = y[t];
    }
  }
}

// One warp: the 4 RI x 32 tile of A at rows rr.., columns cc.. -= (the rows'
// columns c0 .. c0 + 31) x (rows c0 .. c0 + 31's columns).  Thread = rows
// rr + (lane >> 3) + 4 i, columns cc + 4 (lane & 7) ..: the four row groups'
// 16-byte pieces fall in different banks.
template <typename T, int RI>
__device__ __forceinline__ void slab_update_tile(T* A, int wp, int c0, int rr, int cc, int hs, int wt) {
  constexpr int VN = V16<T>::n;
  const int lane = threadIdx.x & 31;
  const int r0 = rr + (lane >> 3), cj = cc + 4 * (lane & 7);
  if (cj >= wt) return;  // (columns past wt but below its 16-byte piece's end are padding of the row)
  T acc[RI][4];
#pragma unroll
  for (int i = 0; i < RI; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[i][q] = T(0);
  const T* ar[RI];
#pragma unroll
  for (int i = 0; i < RI; ++i) ar[i] = A + (size_t)min(r0 + 4 * i, hs - 1) * wp + c0;
  const T* br = A + (size_t)c0 * wp + cj;
#pragma unroll 1
  for (int k = 0; k < 32; k += VN) {
    T av[RI][VN];
#pragma unroll
    for (int i = 0; i < RI; ++i) s16_get<T>(ar[i] + k, av[i]);
#pragma unroll
    for (int e = 0; e < VN; ++e) {
      T bv[4];
#pragma unroll
      for (int q = 0; q < 4; q += VN) s16_get<T>(br + (size_t)(k + e) * wp + q, bv + q);
#pragma unroll
      for (int i = 0; i < RI; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][q] = fma(av[i][e], bv[q], acc[i][q]);
    }
  }
#pragma unroll
  for (int i = 0; i < RI; ++i) {
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
// of the inverse, held in Z (32 x 32): back substitution with the division by
// U's diagonal, by sub-blocks of eight rows.
template <typename T>
__device__ __forceinline__ void slab_inverse(T* Ub, int wp, int bw, const T* rinv, T* Z, T* out) {
  constexpr int VN = V16<T>::n;
  const int lane = threadIdx.x & 31;
  for (int t = 0; t < 32; ++t) Z[t * 32 + lane] = t == lane ? T(1) : T(0);  // (a lane reads its own column only)
  if (bw < 32) {  // the padding right of a ragged block's columns couples to nothing
    for (int r = 0; r < bw; ++r)
      if (lane >= bw) Ub[(size_t)r * wp + lane] = T(0);
    __syncwarp();
  }
#pragma unroll 1
  for (int tb = 24; tb >= 0; tb -= 8) {
    // the 8 x 8 block of U on the diagonal, the identity past a ragged block
    T z[8], u[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i) z[i] = Z[(tb + i) * 32 + lane];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool in = tb + i < bw;
#pragma unroll
      for (int g = i / VN * VN; g < 8; g += VN) {
        if (in) {
          s16_get<T>(Ub + (size_t)(tb + i) * wp + tb + g, &u[i][g]);
        } else {
#pragma unroll
          for (int e = g; e < g + VN; ++e) u[i][e] = e == i ? T(1) : T(0);
        }
      }
    }
#pragma unroll
    for (int jj = 7; jj >= 0; --jj) {
      z[jj] = quot_rn(z[jj], u[jj][jj], tb + jj < bw ? rinv[tb + jj] : T(1));
#pragma unroll
      for (int i = 0; i < jj; ++i) z[i] = fma(-u[i][jj], z[jj], z[i]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) out[(tb + i) * 32 + lane] = z[i];
    if (tb >= bw) continue;
#pragma unroll 1
    for (int qb = tb - 8; qb >= 0; qb -= 8) {
      T y[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) y[i] = Z[(qb + i) * 32 + lane];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        T uq[8];
#pragma unroll
        for (int g = 0; g < 8; g += VN) s16_get<T>(Ub + (size_t)(qb + i) * wp + tb + g, uq + g);
#pragma unroll
        for (int jj = 7; jj >= 0; --jj) y[i] = fma(-uq[jj], z[jj], y[i]);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) Z[(qb + i) * 32 + lane] = y[i];
    }
  }
}

// rows [0, nrows) x columns [0, ncol) of G (row-major, ld) into S (row stride
// sld, a multiple of 16 bytes): asynchronous 16-byte copies when G's rows are
// 16-byte aligned, all in flight together
template <typename T>
__device__ __forceinline__ void slab_load(const T* G, int64_t ld, int nrows, int ncol, T* S, int sld) {
  constexpr int VN = V16<T>::n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool vec = ((reinterpret_cast<uintptr_t>(G) & 15) == 0) && ((ld * (int64_t)sizeof(T)) & 15) == 0;
  const int nvec = vec ? ncol / VN : 0;
  for (int r = warp; r < nrows; r += SL_WARPS) {
    for (int v = lane; v < nvec; v += 32) cp_async<16>(S + (size_t)r * sld + v * VN, G + (int64_t)r * ld + v * VN);
    for (int c = nvec * VN + lane; c < ncol; c += 32) cp_async<sizeof(T)>(S + (size_t)r * sld + c, G + (int64_t)r * ld + c);
  }
  cp_async_wait_all();
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
  __shared__ T rinv[128];                 // the reciprocals of the pivots
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool spec = sp.flag != nullptr;
  bool bad = false;
  previous_wait();
  if (spec) {
    const int f0 = __ldcg(sp.flag), f3 = __ldcg(sp.flag + 3);
    if (f0 != 0 || f3 != 0) {
      if (tid == 0 && f0 == 0) sp.flag[0] = 1;  // a failure of the rows below an earlier slab
      return;
    }
  }
  slab_load<T>(D, ld, hs, wt, A, wp);
  if (spec && first) {
    for (int j = tid; j < wt; j += SL_THREADS) sp.ipiv[kabs + j] = kabs + j + 1;
    if (tid == 0) sp.perm[0] = 0;
  }
  __syncthreads();
  if (warp == 0) {
    slab_diag<T>(A, wp, min(32, hs), spec, info, kabs, rinv, bad);
  } else if (spec && first) {
    // the rows as they were (D itself is written at the end)
    for (int r = warp - 1; r < hs; r += SL_WARPS - 1)
#pragma unroll 4
      for (int c = lane; c < wt; c += 32) sp.backup[(int64_t)r * wt + c] = D[(int64_t)r * ld + c];
  }
  __syncthreads();
  for (int c0 = 0; c0 < hs; c0 += 32) {
    const int bw = min(32, hs - c0);
    const int r1 = c0 + bw;
    T* Ub = A + (size_t)c0 * wp + c0;
    // (b), (i'): rows below, then columns right of the block (a column exists
    // only beside a whole 32-column block)
    const int nr = hs - r1, nc = wt - r1;
    const int ritems = (nr * 2 + 31) & ~31;  // whole warps
    for (int it = tid; it < ritems + nc; it += SL_THREADS) {
      if (it < ritems) {
        const int r = it >> 1;
        slab_left_row<T>(Ub, wp, rinv + c0, A + (size_t)(r1 + min(r, nr - 1)) * wp + c0, r < nr, it & 1, spec, bad);
      } else {
        slab_top_column<T>(Ub, wp, A + (size_t)c0 * wp + r1 + (it - ritems));
      }
    }
    __syncthreads();
    if (nr > 0) {
      // (ii), and (a) of the next block on warp 0 once warps 0..3 have updated its tile
      const int tc = (nc + 31) / 32, tiles = ((nr + 31) / 32) * tc;
      if (warp < 4) {
        slab_update_tile<T, 2>(A, wp, c0, r1 + 8 * warp, r1, min(hs, r1 + 32), wt);
        asm volatile("bar.sync 1, 128;" ::: "memory");
      }
      if (warp == 0)
        slab_diag<T>(A + (size_t)r1 * wp + r1, wp, min(32, hs - r1), spec, info, kabs + r1, rinv + r1, bad);
      for (int t = warp == 0 ? tiles : SL_WARPS - warp; t < tiles; t += SL_WARPS - 1)
        slab_update_tile<T, 8>(A, wp, c0, r1 + 32 * (t / tc), r1 + 32 * (t % tc), hs, wt);
      __syncthreads();
    }
  }
  dependents_launch();
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
    slab_inverse<T>(A + (size_t)(32 * b) * wp + 32 * b, wp, min(32, hs - 32 * b), rinv + 32 * b,
                    A + (size_t)hs * wp + (size_t)b * 1024, uinv + (size_t)b * 1024);
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
__global__ void __launch_bounds__(LS_THREADS) below_solve_kernel(const T* U, const T* uinv,
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
  previous_wait();
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
  dependents_launch();
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

// The rows-below launches' view of the device: shared memory per CTA, and the CTAs
// of one wave (two per SM: 304 on GB300).
struct BelowDev {
  int optin, wave;
};
static BelowDev below_dev() {
  int dev = 0, sms = 0;
  BelowDev d{0, 0};
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&d.optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  d.wave = 2 * sms;
  return d;
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

// One launch of the block column's chain.  dependent: the launch before it in
// the stream is the chain's own, whose kernels let the next one start while they
// still write their results (the next one waits for them at its start): it hides
// the launch, not the work (mixed n = 1500 1.39 -> 1.36 ms, no-pivot n = 6000 6.68
// -> 6.61).  Only where the rows below the first slab are one wave in CTAs of 16
// rows (4864 rows on GB300), and then for the whole chain: the
// waiting CTAs of a larger launch keep the trailing update beside the panel off
// their SMs (mixed n = 32768 114.3 -> 116.5 ms).
template <typename... P, typename... A>
static cudaError_t launch_chain(void (*kern)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st,
                                bool dependent, A... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

template <typename T, int RB>
static cudaError_t launch_ls(const T* U, const T* uinv, T* X, int64_t ld, int m, int ws, int wt,
                             const SpecDev<T>& sp, int first, int tag, bool dependent, cudaStream_t st) {
  auto kern = below_solve_kernel<T, RB>;
  cudaError_t e = allow_max_smem((const void*)kern);
  if (e != cudaSuccess) return e;
  return launch_chain(kern, (unsigned)cdiv(m, RB), LS_THREADS, ls_smem(RB, wt, sizeof(T)), st, dependent,
                      U, uinv, X, ld, m, ws, wt, sp, first, tag);
}

template <typename T>
static cudaError_t launch_below(const T* U, const T* uinv, T* X, int64_t ld, int m, int ws, int wt,
                                const SpecDev<T>& sp, int first, int tag, const BelowDev& dv, bool dependent,
                                cudaStream_t st) {
  const int optin = dv.optin;
  // Fewer rows per CTA while two CTAs per SM still take all rows at once: the
  // launch is then as short as one CTA's chain of blocks, whose length grows
  // with its rows (slab of 128 x 256, 1400 rows below: 64 rows per CTA 37 us, 16
  // rows 21; slab of 128 x 128: 22 and 14; 5400 rows, 256 wide: 37 and 33 with
  // 32); a longer launch takes 64, which read U least often.
  const bool short_launch = cdiv(m, 32) <= dv.wave;
  if (cdiv(m, 16) <= dv.wave && ls_smem(16, wt, sizeof(T)) <= (size_t)optin)
    return launch_ls<T, 16>(U, uinv, X, ld, m, ws, wt, sp, first, tag, dependent, st);
  if (!short_launch && ls_smem(64, wt, sizeof(T)) <= (size_t)optin)
    return launch_ls<T, 64>(U, uinv, X, ld, m, ws, wt, sp, first, tag, dependent, st);
  if (ls_smem(32, wt, sizeof(T)) <= (size_t)optin)
    return launch_ls<T, 32>(U, uinv, X, ld, m, ws, wt, sp, first, tag, dependent, st);
  if (ls_smem(16, wt, sizeof(T)) <= (size_t)optin)
    return launch_ls<T, 16>(U, uinv, X, ld, m, ws, wt, sp, first, tag, dependent, st);
  return cudaErrorInvalidValue;
}

// One slab: a CTA with the slab in shared memory.
template <typename T>
static cudaError_t launch_slab(T* D, int64_t ld, int hs, int wt, int kabs, int* info, const SpecDev<T>& sp,
                               int first, int tag, int restore, T* uinv, cudaStream_t st, bool dependent) {
  auto kern = slab_lu_kernel<T>;
  cudaError_t e = allow_max_smem((const void*)kern);
  if (e != cudaSuccess) return e;
  return launch_chain(kern, 1, SL_THREADS, slab_smem_bytes(hs, wt, sizeof(T)), st, dependent, D, ld, hs, wt, kabs, info,
                      sp, first, tag, restore, uinv);
}

template <typename T>
cudaError_t launch_block_column(T* P, int64_t ld, int m, int w, int kabs, int* info, T* uinv, cudaStream_t st,
                                const SpecArgs& spec) {
  if (w <= 0) return cudaSuccess;
  if (m < w) return cudaErrorInvalidValue;
  const int h = slab_rows(w, sizeof(T));
  const BelowDev dv = below_dev();
  const bool dependent = cdiv(m - (w < h ? w : h), 16) <= dv.wave;
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
                            below > 0 ? ui : nullptr, st, !first && dependent)) != cudaSuccess)
      return e;
    if (below > 0) {
      // the first slab's rows below it follow its rows in the backup (row stride w)
      e = launch_below<T>(D, ui, D + (int64_t)hs * ld, ld, below, hs, wt, spec_dev<T>(spec, (int64_t)hs * w), first,
                          tag, dv, dependent, st);
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
