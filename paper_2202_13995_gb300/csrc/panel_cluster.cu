// Panel factorization with partial pivoting, the panel resident in shared
// memory: on one thread-block cluster, and for panels that 16 CTAs do not hold
// or that keep more FP64 pipes busy, on the whole grid (at the end).
//
// The same computation as panel_getrf_kernel (the paper's diagonal and left
// blocks of a block iteration, factored together because partial pivoting
// searches every row below the diagonal; arxiv 2202.13995, section "Base
// Implementation"): for each column j, p = the first row of largest |a| at or
// below j, swap rows j and p, divide the entries below the diagonal by the
// pivot, rank-1 update of the columns to the right.
//
// The grid is one cluster of CL <= 16 CTAs; CTA c holds the panel rows
// [c R, c R + R), all w columns, in shared memory for the whole panel.  Rows do
// not move: every row carries its current position (pos), a pivot swaps two
// positions, and at the end each row is written to its position.
//
// What bounds it is the chain of w columns, one exchange of candidates each:
//  - every CTA sends its best (|a|, position), the pivot's reciprocal and the
//    row's values right of the diagonal into every peer's shared memory
//    (st.async, whose bytes complete a transaction barrier there): one hop
//    through distributed shared memory, no grid barrier and no L2 round trip;
//  - what the exchange needs of column j + 1 comes first (the multipliers of
//    column j, column j + 1's update and search, the candidate row's values);
//    the update of the other columns runs while the candidates travel;
//  - the warps have roles: those of the chain (one per 32 rows) read the
//    records and take the multipliers, the next two columns and the search, the
//    others update the rest, so the FP64 pipes work through the chain's waits
//    (all warps in step: 2.5 us a column of 512 x 64, 2.9 of 1024 x 128).
// Quotients come from the pivot's reciprocal by P. Markstein's correction
// (see quot_rn), three multiply-adds instead of a division: GB300 issues an
// FP64 warp instruction once in 64 cycles per SM quarter, and a division takes
// nine of them.
// Measured (us per column, step call, cooperative kernel -> this one): FP64
// 512 x 64 5.1 -> 2.0, 1023 x 64 5.5 -> 2.4, 1024 x 128 5.5 -> 2.7; FP32
// 512 x 64 3.6 -> 1.6, 2500 x 128 4.0 -> 1.6, 6000 x 64 4.3 -> 2.2.
//
// A record's buffer is reused every third column: its pivot row is read until
// a CTA has finished column j, a peer sends column j + 3 only after it has
// this CTA's record of column j + 2, and that is sent after column j is done.
//
// Every wait on a transaction barrier is bounded; a CTA whose wait runs out
// raises ST_TIMEOUT and goes to the closing cluster barrier, which all CTAs
// reach (the others' waits run out too).
#include <climits>
#include <mutex>

#include "common.cuh"
#include "kernels.h"
#include "panel_wait.cuh"
#include "tc_ptx.cuh"

namespace gb {

constexpr int PC_CLMAX = 16;
constexpr int PC_NTMAX = 512;
constexpr int PC_NBUF = 3;

template <typename T>
struct PcParams {
  T* A;  // W(k, k)
  int64_t ld;
  int m, w, R;
  int kabs;
  int* ipiv;
  int* info;
  int* status;
  int* perm;
};

// A candidate's record: 16-byte pieces, the header first (key, position,
// reciprocal), then the row's w values.  Column j's record is sent from the
// piece that holds column j on.
template <typename T>
struct PcRec;
template <>
struct PcRec<double> {
  static constexpr int VN = 2, HC = 2;  // values per piece, header pieces
};
template <>
struct PcRec<float> {
  static constexpr int VN = 4, HC = 1;
};

__host__ __device__ inline int pc_pieces(int w, int tsize) {
  return (tsize == 8 ? PcRec<double>::HC : PcRec<float>::HC) + (w * tsize + 15) / 16;
}
// the tile, the records (received ones and the CTA's own; they hold at least
// R positions at the end)
__host__ __device__ inline size_t pc_smem_bytes(int R, int w, int cl, int tsize) {
  const size_t tile = ((size_t)w * (R | 1) * tsize + 15) / 16 * 16;
  const size_t recs = (size_t)(PC_NBUF * cl + 1) * pc_pieces(w, tsize) * 16;
  return tile + (recs > (size_t)R * 4 ? recs : (size_t)R * 4);
}

// Pivot-search order as unsigned words: larger first, 0 = no candidate (a
// magnitude's bit pattern is below 0x7ff00001 / 0x7f800001).
struct PcKey {
  unsigned hi, lo;
  int pos;
};
__device__ __forceinline__ PcKey pc_key(float v, bool valid, int pos) {
  return {valid ? __float_as_uint(pivot_mag(v)) + 1u : 0u, 0u, valid ? pos : INT_MAX};
}
__device__ __forceinline__ PcKey pc_key(double v, bool valid, int pos) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(pivot_mag(v));
  return {valid ? (unsigned)(b >> 32) + 1u : 0u, valid ? (unsigned)b : 0u, valid ? pos : INT_MAX};
}
__device__ __forceinline__ bool pc_better(const PcKey& a, const PcKey& b) {
  if (a.hi != b.hi) return a.hi > b.hi;
  if (a.lo != b.lo) return a.lo > b.lo;
  return a.pos < b.pos;
}
// the best key of the warp in every lane; true in the lane that holds it
// (positions are distinct, so at most one lane does)
template <typename T>
__device__ __forceinline__ bool pc_warp_best(PcKey& k) {
  const unsigned mh = __reduce_max_sync(0xffffffffu, k.hi);
  bool in = k.hi == mh;
  unsigned ml = 0u;
  if (sizeof(T) == 8) {
    ml = __reduce_max_sync(0xffffffffu, in ? k.lo : 0u);
    in = in && k.lo == ml;
  }
  const int mp = (int)__reduce_min_sync(0xffffffffu, in ? (unsigned)k.pos : (unsigned)INT_MAX);
  const bool mine = in && k.pos == mp && mh != 0u;
  k = {mh, ml, mp};
  return mine;
}

// 16 bytes into a peer's shared memory, counted on the peer's transaction
// barrier (both shared::cluster addresses of the same CTA)
__device__ __forceinline__ void pc_send16(uint32_t dst, longlong2 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];" ::"r"(dst),
               "l"(v.x), "l"(v.y), "r"(bar)
               : "memory");
}

// A CTA's rows (at A, row stride ld) to shared memory, four of a warp's rows in
// flight at a time
template <typename T>
__device__ __forceinline__ void pc_load_rows(T* S, int Rs, const T* A, int64_t ld, int rows, int w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int rb = warp; rb < rows; rb += 4 * nw) {
    for (int c = lane; c < w; c += 32) {
      T x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int rr = rb + i * nw;
        x[i] = rr < rows ? __ldcg(A + (int64_t)rr * ld + c) : T(0);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int rr = rb + i * nw;
        if (rr < rows) S[(size_t)c * Rs + rr] = x[i];
      }
    }
  }
}

// ... and back, row rr to position sp[rr] of the panel at A
template <typename T>
__device__ __forceinline__ void pc_store_rows(T* A, int64_t ld, const T* S, int Rs, const int* sp, int rows, int w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int rr = warp; rr < rows; rr += nw) {
    T* dst = A + (int64_t)sp[rr] * ld;
    for (int c = lane; c < w; c += 32) dst[c] = S[(size_t)c * Rs + rr];
  }
}

// Columns c, c + step, .. below w of this lane's row (at Sr, column stride Rs) -= l
// times the pivot row
template <typename T>
__device__ __forceinline__ void pc_update(T* Sr, int Rs, const T* pr, T l, int c, int step, int w) {
  const size_t st = (size_t)step * Rs;
  T* x = Sr + (size_t)c * Rs;
  for (; c + 3 * step < w; c += 4 * step, x += 4 * st) {
    T v[4], u[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[q] = x[q * st];
      u[q] = pr[c + q * step];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q * st] = fma(-l, u[q], v[q]);
  }
  T v[3], u[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (c + q * step < w) {
      v[q] = x[q * st];
      u[q] = pr[c + q * step];
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q)
    if (c + q * step < w) x[q * st] = fma(-l, u[q], v[q]);
}

template <typename T>
__global__ void __launch_bounds__(PC_NTMAX, 1) panel_cluster_kernel(PcParams<T> P) {
  constexpr int VN = PcRec<T>::VN, HC = PcRec<T>::HC;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long bars[PC_NBUF];
  __shared__ uint4 red[PC_NTMAX / 32];  // each row group's best: key, position, row
  __shared__ int sel[2];  // the current column's pivot: position, CTA
  __shared__ int abort_flag;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  const int cta = (int)cluster_rank(), CL = (int)gridDim.x;
  const int R = P.R, w = P.w, Rs = R | 1;
  const int64_t ld = P.ld;
  const int row0 = cta * R;
  const int rloc = max(0, min(P.m, row0 + R) - row0);
  // A warp serves one group of 32 rows, a lane per row.  Class 0 of the group's
  // warps takes the chain: the records, the multipliers, the next two columns,
  // the search.  The other classes update the other columns meanwhile; they
  // learn of the pivot at the barrier that ends the search.  (A CTA of so many
  // rows that every warp is a chain warp updates them itself.)
  const int RG = (R + 31) / 32;
  const int NC = nw / RG;  // classes; warps past NC * RG only help with the records
  const int rg = warp % RG, cls = warp / RG;
  const int r = rg * 32 + lane;
  const bool live = cls < NC && r < rloc;
  const bool chain = warp < RG;
  const bool all_upd = NC == 1;
  const int c_off = all_upd ? 3 + cls : 2 + cls, c_step = all_upd ? NC : NC - 1;  // columns j + c_off, + c_step, ..
  const bool upd = cls < NC && (all_upd || !chain);
  const int pieces = pc_pieces(w, sizeof(T));
  const size_t tile = ((size_t)w * Rs * sizeof(T) + 15) / 16 * 16;
  T* S = reinterpret_cast<T*>(smem_raw);  // [w][Rs]: column c of the tile, row r
  unsigned char* recs = smem_raw + tile;  // [PC_NBUF][CL][pieces][16]
  unsigned char* mine = recs + (size_t)PC_NBUF * CL * pieces * 16;  // this CTA's own record
  T* mrow = reinterpret_cast<T*>(mine + 16 * HC);
  T* Sr = S + r;  // this lane's row (dereferenced by live lanes only)

  if (tid == 0) {
    for (int b = 0; b < PC_NBUF; ++b) mbar_init(smem_u32(&bars[b]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    abort_flag = 0;
    if (cta == 0) P.perm[0] = 0;
  }
  pc_load_rows(S, Rs, P.A + (int64_t)row0 * ld, ld, rloc, w);
  __syncthreads();
  cluster_sync();  // every peer's barriers are set up, and the count of perm is zero

  // this warp's peers (at most two) and this CTA's record in them
  const uint32_t bar0 = smem_u32(&bars[0]);
  const uint32_t dst0 = smem_u32(recs + (size_t)cta * pieces * 16);
  const uint32_t bufstep = (uint32_t)(CL * pieces * 16);
  uint32_t pbar[2], pdst[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int peer = warp + i * nw;
    pbar[i] = cluster_map(bar0, (uint32_t)(peer < CL ? peer : 0));
    pdst[i] = cluster_map(dst0, (uint32_t)(peer < CL ? peer : 0));
  }

  int pos = row0 + r;  // this lane's row's position
  bool act = live;     // ... and whether the row is below the current column's diagonal
  // column j's pivot moved to row j: positions p and j change places
  auto move = [&](int j, int p) {
    if (live) {
      if (pos == p)
        pos = j;
      else if (pos == j)
        pos = p;
    }
    act = live && pos > j;
  };
  // The CTA's candidate of column c (key `best` of this lane's row, chain
  // warps): its record to every peer.  With c > 0 the columns right of c still
  // lack their update by column c - 1, whose pivot row (sel) pr is set to.
  auto publish = [&](int c, int buf, int pbuf, PcKey best, const T*& pr) {
    if (chain) {
      const bool own = pc_warp_best<T>(best);
      const unsigned at = __ballot_sync(0xffffffffu, own);
      if (lane == 0) red[warp] = make_uint4(best.hi, best.lo, (unsigned)best.pos, (unsigned)(rg * 32 + __ffs(at) - 1));
    }
    __syncthreads();
    if (abort_flag) return false;
    if (c > 0) {
      pr = reinterpret_cast<const T*>(recs + (size_t)pbuf * CL * pieces * 16 + (size_t)sel[1] * pieces * 16 + 16 * HC);
      if (!chain) move(c - 1, sel[0]);
    }
    uint4 e = red[lane < RG ? lane : 0];
    if (RG > 1) {
      PcKey k{lane < RG ? e.x : 0u, lane < RG ? e.y : 0u, lane < RG ? (int)e.z : INT_MAX};
      const bool own = pc_warp_best<T>(k);
      const unsigned at = __ballot_sync(0xffffffffu, own);
      e.w = __shfl_sync(0xffffffffu, e.w, at ? __ffs(at) - 1 : 0);
      e.x = k.hi;
      e.y = k.lo;
      e.z = (unsigned)k.pos;
    }
    const bool any = e.x != 0u;
    if (any) {
      const T* Sk = S + e.w;
      const T lc = c > 0 ? Sk[(size_t)(c - 1) * Rs] : T(0);
      for (int q = c + tid; q < w; q += nt) {
        T v = Sk[(size_t)q * Rs];
        if (c > 0 && q > c) v = fma(-lc, pr[q], v);
        mrow[q] = v;
      }
    }
    if (warp == nw - 1) {
      const T rv = recip_rn(any ? S[(size_t)c * Rs + e.w] : T(0));
      if (lane == 0) {
        unsigned* h = reinterpret_cast<unsigned*>(mine);
        h[0] = e.x;
        h[1] = e.z;
        if (sizeof(T) == 8) h[2] = e.y;
        reinterpret_cast<T*>(mine)[2] = rv;
      }
    }
    __syncthreads();
    const int p0 = HC + c / VN;  // row pieces from column c's on
    const int np = HC + pieces - p0;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (warp + i * nw < CL) {
        const uint32_t bar = pbar[i] + 8u * (uint32_t)buf, dst = pdst[i] + bufstep * (uint32_t)buf;
        for (int x = lane; x < np; x += 32) {
          const int pc = x < HC ? x : p0 + x - HC;
          pc_send16(dst + 16u * (uint32_t)pc, reinterpret_cast<const longlong2*>(mine)[pc], bar);
        }
      }
    }
    return true;
  };
  // arm the barrier of column c's records (its previous phase is complete)
  auto arm = [&](int c, int buf) {
    if (tid == 0) mbar_expect_tx(bar0 + 8u * (uint32_t)buf, (uint32_t)(CL * (pieces - c / VN) * 16));
  };

  T cur = live ? Sr[0] : T(0);                                    // chain warps: column j of the row,
  T nxt = live && w > 1 ? Sr[(size_t)Rs] : T(0);                  // and column j + 1 before column j's update
  const T* pr = nullptr;
  arm(0, 0);
  bool ok = publish(0, 0, 0, pc_key(cur, live, pos), pr);
  int buf = 0;
  uint32_t par = 0;
  for (int j = 0; j < w && ok; ++j) {
    const int nbuf = buf + 1 == PC_NBUF ? 0 : buf + 1;
    PcKey best{0u, 0u, INT_MAX};
    if (chain) {
      const uint32_t bar = bar0 + 8u * (uint32_t)buf;
      pc_wait(bar, par, &abort_flag, P.status);
      __syncwarp();
      if (j + 1 < w) arm(j + 1, nbuf);
      // the pivot: the best of the CTAs' candidates
      const unsigned char* rb = recs + (size_t)buf * bufstep;
      PcKey k{0u, 0u, INT_MAX};
      if (lane < CL) {
        const unsigned* h = reinterpret_cast<const unsigned*>(rb + (size_t)lane * pieces * 16);
        k = {h[0], sizeof(T) == 8 ? h[2] : 0u, (int)h[1]};
      }
      const bool kown = pc_warp_best<T>(k);
      const unsigned bal = __ballot_sync(0xffffffffu, kown);
      const int win = bal ? __ffs(bal) - 1 : 0;
      const unsigned char* rec = rb + (size_t)win * pieces * 16;
      pr = reinterpret_cast<const T*>(rec + 16 * HC);  // the pivot row, columns j .. w
      const T rinv = reinterpret_cast<const T*>(rec)[2];
      const T piv = pr[j];
      const T u1 = j + 1 < w ? pr[j + 1] : T(0);
      if (!GB_IN_BOUNDS(P.status, k.hi == 0u || (k.pos >= j && k.pos < P.m))) k.pos = j;
      if (tid == 0) {
        sel[0] = k.pos;
        sel[1] = win;
        if (cta == 0) {
          P.ipiv[P.kabs + j] = P.kabs + k.pos + 1;
          if (!nonzero(piv)) atomicMin(P.info, P.kabs + j + 1);
          if (is_inf_mag(pivot_mag(piv))) atomicOr(P.status, ST_RANGE);  // a non-finite candidate
        }
      }
      move(j, k.pos);
      // multipliers, column j + 1 and its search
      if (act) {
        const T l = nonzero(piv) ? quot_rn(cur, piv, rinv) : cur;
        Sr[(size_t)j * Rs] = l;
        cur = fma(-l, u1, nxt);
        if (j + 1 < w) {
          Sr[(size_t)(j + 1) * Rs] = cur;
          best = pc_key(cur, true, pos);
        }
      }
    }
    if (j + 1 == w) break;
    ok = publish(j + 1, nbuf, buf, best, pr);
    if (!ok) break;
    // while the candidates travel: column j + 2, which the chain needs next,
    // by the chain warps, the columns after it by the others
    if (act) {
      const T l = Sr[(size_t)j * Rs];
      if (chain && j + 2 < w) {
        T* x = Sr + (size_t)(j + 2) * Rs;
        nxt = fma(-l, pr[j + 2], x[0]);
        x[0] = nxt;
      }
      if (upd) pc_update(Sr, Rs, pr, l, j + c_off, c_step, w);
    }
    buf = nbuf;
    if (buf == 0) par ^= 1u;
  }
  __syncthreads();
  if (!abort_flag) {
    // each row to its position; the rows that moved to the permutation record
    int* sp = reinterpret_cast<int*>(recs);  // [R] (the records are all read)
    if (chain && live) sp[r] = GB_IN_BOUNDS(P.status, pos >= 0 && pos < P.m) ? pos : row0 + r;
    __syncthreads();
    pc_store_rows(P.A, ld, S, Rs, sp, rloc, w);
    if (chain && live && pos != row0 + r) {
      const int q = atomicAdd(P.perm, 1);
      if (GB_IN_BOUNDS(P.status, q < 2 * w)) {
        P.perm[1 + q] = pos;
        P.perm[1 + 2 * w + q] = row0 + r;
      }
    }
  } else {
    // records may still be on their way to a CTA whose wait ran out
    const uint64_t t0 = gtimer();
    while (gtimer() - t0 < 1000000ull) __nanosleep(1000);
  }
  cluster_sync();  // no CTA leaves while a peer may still send to it
}

// CTAs of a panel's cluster: rows of 32 (FP64: the FP64 pipes of as many SMs as
// help) or 64 (FP32) per CTA up to 16 CTAs; -1 when the tile does not fit the
// shared memory then.  grid: the grid form can take the panel instead, which an
// FP64 panel of m w > 100,000 is faster on, bound as it is by the FP64 pipes of
// 16 SMs (us, cluster and grid: 1500 x 64 167 and 180, 2048 x 64 188 and 178,
// 2048 x 32 96 and 105, 3000 x 32 102 and 103, 4096 x 32 117 and 102, 1024 x 128
// 348 and 341); without it the line is the cooperative kernel's, 360,000
// (3000 x 128: 6.1 and 6.0 us a column).
static int pc_config(int m, int w, int tsize, int optin, bool grid, int* R, int* nt, size_t* smem) {
  if (w < 1 || w > 512 || m < w) return -1;
  const int target = tsize == 8 ? 32 : 64;
  int cl = 1;
  while (cl < PC_CLMAX && cl * target < m) cl *= 2;
  *R = (int)cdiv(m, cl);
  *nt = *R <= target ? 256 : PC_NTMAX;  // (a warp per 32 rows at least)
  if (*R > PC_NTMAX) return -1;
  *smem = pc_smem_bytes(*R, w, cl, tsize);
  if (*smem + 1024 > (size_t)optin) return -1;
  if (tsize == 8 && (int64_t)m * w > (grid ? 100000 : 360000)) return -1;
  return cl;
}

template <typename T>
static cudaLaunchConfig_t pc_launch(int cl, int nt, size_t smem, cudaStream_t st, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cl);
  cfg.blockDim = dim3(nt);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = cl;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

template <typename T>
static cudaError_t pc_prepare() {
  cudaError_t e = allow_max_smem((const void*)panel_cluster_kernel<T>);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute((const void*)panel_cluster_kernel<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

// Whether the panel fits the cluster kernel and such a cluster can be placed
// on the current device (asked of the runtime once per cluster and block size,
// with the largest shared memory).
template <typename T>
bool panel_cluster_fits(int m, int w, const DevInfo& dev, bool grid) {
  int R = 0, nt = 0;
  size_t smem = 0;
  const int cl = pc_config(m, w, sizeof(T), dev.max_smem_optin, grid, &R, &nt, &smem);
  if (cl < 0) return false;
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess || device < 0 || device >= 64) return false;
  static std::mutex mu;
  static signed char known[64][2][PC_CLMAX + 1] = {};  // 0 unknown, 1 yes, -1 no
  std::lock_guard<std::mutex> lk(mu);
  signed char& kn = known[device][nt == PC_NTMAX][cl];
  if (kn == 0) {
    int n = 0;
    cudaLaunchAttribute at[1];
    cudaFuncAttributes fa;
    cudaError_t e = pc_prepare<T>();
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, (const void*)panel_cluster_kernel<T>);
    if (e == cudaSuccess) {
      cudaLaunchConfig_t cfg =
          pc_launch<T>(cl, nt, (size_t)dev.max_smem_optin - fa.sharedSizeBytes, nullptr, at);
      e = cudaOccupancyMaxActiveClusters(&n, (const void*)panel_cluster_kernel<T>, &cfg);
    }
    if (e != cudaSuccess) cudaGetLastError();
    kn = (e == cudaSuccess && n > 0) ? 1 : -1;
  }
  return kn > 0;
}

template <typename T>
cudaError_t launch_panel_cluster(T* Wkk, int64_t ldw, int m, int w, int kabs, int* ipiv, int* info, int* status,
                                 int* perm, const DevInfo& dev, cudaStream_t st) {
  PcParams<T> P;
  int nt = 0;
  size_t smem = 0;
  const int cl = pc_config(m, w, sizeof(T), dev.max_smem_optin, false, &P.R, &nt, &smem);
  if (cl < 0) return cudaErrorInvalidConfiguration;
  cudaError_t e = pc_prepare<T>();
  if (e != cudaSuccess) return e;
  P.A = Wkk;
  P.ld = ldw;
  P.m = m;
  P.w = w;
  P.kabs = kabs;
  P.ipiv = ipiv;
  P.info = info;
  P.status = status;
  P.perm = perm;
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = pc_launch<T>(cl, nt, smem, st, at);
  return cudaLaunchKernelEx(&cfg, panel_cluster_kernel<T>, P);
}

// ============================================================ the same on the whole grid
// Panels too large for one cluster: the CTAs of a cooperative launch hold R
// rows each, all columns, in shared memory, and work as above; only the
// exchange differs.  A CTA's record lies in global memory: a 16-byte header
// (key and position) and the row beside it.  Every 8-byte word of either
// carries the column's stamp next to its data, so readers know a word by
// itself and no fence orders the stores (a release store that waits for the
// row's stores cost 1 us a column).  Every CTA polls all headers, picks the
// pivot and reads its row once: two L2 round trips a column, with the update of
// the other columns under them.  Against the kernel in
// panel.cu (a counter barrier, every candidate row read by every CTA,
// sub-panels of 32 columns written back, interchanged and updated through L2)
// no value but the pivot row crosses L2 twice.
// Measured (us per column, that kernel -> this one): FP64 6000 x 64 5.9 -> 3.3,
// 8192 x 128 6.7 -> 3.1, 7000 x 256 7.7 -> 3.6 (there the FP64 pipes set the
// pace: 256 columns of 47 rows); FP32 8192 x 128 4.5 -> 2.2.
// The record buffers' stamps are cleared before the launch; a buffer is
// reused every third column (the argument above).  What is not stamped, the rows
// that a CTA loads before its first header and others overwrite at the end and the
// count of the permutation record, is ordered once a panel: the thread that writes
// the headers fences before its first one, every thread after the last column,
// when its CTA has read every CTA's first header.  Every poll is bounded; a CTA
// whose poll runs out raises ST_TIMEOUT and leaves, and so do the others in their
// turn.

template <typename T>
struct PrParams {
  T* A;  // W(k, k)
  int64_t ld;
  int m, w, R;
  int kabs;
  int* ipiv;
  int* info;
  int* status;
  int* perm;
  ulonglong2* head;  // [PC_NBUF][G]
  typename PrWord<T>::type* rows;  // [PC_NBUF][G][rstride]: the row's w values, its reciprocal at w
  int rstride;
};

__host__ __device__ inline size_t pr_smem_bytes(int R, int w, int tsize) {
  const size_t tile = ((size_t)w * (R | 1) * tsize + 15) / 16 * 16;
  return tile + (size_t)PC_NBUF * (w + 1) * tsize + (size_t)R * sizeof(int);
}

constexpr int PR_HL = 5;  // headers per polling lane: up to 160 CTAs
constexpr int PR_RL = 4;  // pivot row values per chain lane in flight

__global__ void __launch_bounds__(PC_NTMAX, 1) panel_grid_f64_kernel(PrParams<double> P) {
  using T = double;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint4 red[PC_NTMAX / 32];   // each row group's best: key, position, row
  __shared__ int sel;  // the current column's pivot: position
  __shared__ int abort_flag;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  const int cta = blockIdx.x, G = gridDim.x;
  const int R = P.R, w = P.w, Rs = R | 1;
  const int64_t ld = P.ld;
  const int row0 = cta * R;
  const int rloc = max(0, min(P.m, row0 + R) - row0);
  // (row groups, classes and chain warps as in panel_cluster_kernel)
  const int RG = (R + 31) / 32;
  const int NC = nw / RG;
  const int rg = warp % RG, cls = warp / RG;
  const int r = rg * 32 + lane;
  const bool live = cls < NC && r < rloc;
  const bool chain = warp < RG;
  const bool all_upd = NC == 1;
  const int c_off = all_upd ? 3 + cls : 2 + cls, c_step = all_upd ? NC : NC - 1;
  const bool upd = cls < NC && (all_upd || !chain);
  const size_t tile = ((size_t)w * Rs * sizeof(T) + 15) / 16 * 16;
  T* S = reinterpret_cast<T*>(smem_raw);
  T* prow = reinterpret_cast<T*>(smem_raw + tile);  // [PC_NBUF][w + 1]: pivot rows
  int* sp = reinterpret_cast<int*>(prow + (size_t)PC_NBUF * (w + 1));  // [R] positions, at the end
  T* Sr = S + r;

  if (tid == 0) {
    abort_flag = 0;
    if (cta == 0) P.perm[0] = 0;
  }
  pc_load_rows(S, Rs, P.A + (int64_t)row0 * ld, ld, rloc, w);
  __syncthreads();

  int pos = row0 + r;
  bool act = live;
  auto move = [&](int j, int p) {
    if (live) {
      if (pos == p)
        pos = j;
      else if (pos == j)
        pos = p;
    }
    act = live && pos > j;
  };
  // this CTA's candidate of column c to global memory (pr: the pivot row of
  // column c - 1, which the columns right of c still lack)
  auto publish = [&](int c, int buf, PcKey best, const T* pr) {
    if (chain) {
      const bool own = pc_warp_best<T>(best);
      const unsigned at = __ballot_sync(0xffffffffu, own);
      if (lane == 0) red[warp] = make_uint4(best.hi, best.lo, (unsigned)best.pos, (unsigned)(rg * 32 + __ffs(at) - 1));
    }
    __syncthreads();
    if (abort_flag) return false;
    if (c > 0 && !chain) move(c - 1, sel);
    uint4 e = red[lane < RG ? lane : 0];
    if (RG > 1) {
      PcKey k{lane < RG ? e.x : 0u, lane < RG ? e.y : 0u, lane < RG ? (int)e.z : INT_MAX};
      const bool own = pc_warp_best<T>(k);
      const unsigned at = __ballot_sync(0xffffffffu, own);
      e.w = __shfl_sync(0xffffffffu, e.w, at ? __ffs(at) - 1 : 0);
      e.x = k.hi;
      e.y = k.lo;
      e.z = (unsigned)k.pos;
    }
    const unsigned stamp = (unsigned)c + 1u;
    if (c == 0 && tid == nt - 1) __threadfence();  // (the CTA's row loads and the count's zero, before the barrier above)
    if (tid == nt - 1)
      pr_store(P.head + (size_t)buf * G + cta,
               make_ulonglong2(((unsigned long long)e.x << 32) | stamp,
                               ((unsigned long long)e.y << 32) | ((e.x ? e.z : 0u) << 12) | stamp));
    if (e.x != 0u) {
      auto* grow = P.rows + (size_t)(buf * G + cta) * P.rstride;
      const T* Sk = S + e.w;
      const T lc = pr != nullptr ? Sk[(size_t)(c - 1) * Rs] : T(0);
      for (int q = c + tid; q < w; q += nt) {
        T v = Sk[(size_t)q * Rs];
        if (pr != nullptr && q > c) v = fma(-lc, pr[q], v);
        PrWord<T>::put(grow + q, v, stamp);
      }
      if (warp == nw - 1) {
        const T rv = recip_rn(Sk[(size_t)c * Rs]);
        if (lane == 0) PrWord<T>::put(grow + w, rv, stamp);
      }
    }
    __syncthreads();  // (the candidate's row is read before its columns are updated)
    return true;
  };
  auto fetch = [&](const typename PrWord<T>::type* q, T& v, unsigned stamp) {
    pr_fetch<T>(q, v, stamp, &abort_flag, P.status);
  };

  T cur = live ? Sr[0] : T(0);
  T nxt = live && w > 1 ? Sr[(size_t)Rs] : T(0);
  bool ok = publish(0, 0, pc_key(cur, live, pos), nullptr);
  int buf = 0;
  for (int j = 0; j < w && ok; ++j) {
    const int nbuf = buf + 1 == PC_NBUF ? 0 : buf + 1;
    const unsigned stamp = (unsigned)j + 1u;
    T* pr = prow + (size_t)buf * (w + 1);
    PcKey best{0u, 0u, INT_MAX};
    if (chain) {
      // every chain warp polls all headers, PR_HL per lane, and picks the pivot
      PcKey k{0u, 0u, INT_MAX};
      int kc = 0;
      {
        ulonglong2 h[PR_HL];
        auto there = [&](const ulonglong2& v) { return (unsigned)v.x == stamp && ((unsigned)v.y & 0xfffu) == stamp; };
        auto all = [&]() {
          bool got = true;
#pragma unroll
          for (int i = 0; i < PR_HL; ++i) {
            const int t = lane + 32 * i;
            if (t < G) {
              h[i] = pr_load(P.head + (size_t)buf * G + t);
              got &= there(h[i]);
            }
          }
          return got;
        };
        if (!all()) {
          const uint64_t t0 = gtimer();
          while (!all()) {
            if (*(volatile int*)&abort_flag) break;
            if (gtimer() - t0 > GB_SPIN_LIMIT_NS) {
              atomicOr(P.status, ST_TIMEOUT);
              *(volatile int*)&abort_flag = 1;  // seen by every thread after the CTA's next barrier
              break;
            }
          }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < PR_HL; ++i) {
          const int t = lane + 32 * i;
          if (t < G) {
            PcKey q;
            q.hi = (unsigned)(h[i].x >> 32);
            q.lo = (unsigned)(h[i].y >> 32);
            q.pos = q.hi ? (int)((unsigned)h[i].y >> 12) : INT_MAX;
            if (pc_better(q, k)) {
              k = q;
              kc = t;
            }
          }
        }
      }
      const bool own = pc_warp_best<T>(k);
      const unsigned at = __ballot_sync(0xffffffffu, own);
      const int win = __shfl_sync(0xffffffffu, kc, at ? __ffs(at) - 1 : 0);
      const auto* grow = P.rows + (size_t)(buf * G + win) * P.rstride;
      // the pivot row: what the chain needs, and the rest to shared memory
      // (read after the next barrier), its loads in flight together
      T piv = T(0), rinv = T(0), u1 = T(0);
      T rest[PR_RL];
      bool got = PrWord<T>::get(grow + j, piv, stamp);
      got &= PrWord<T>::get(grow + w, rinv, stamp);
      if (j + 1 < w) got &= PrWord<T>::get(grow + j + 1, u1, stamp);
      const int q0 = j + 1 + tid, qs = 32 * RG;
      bool gotr = true;
#pragma unroll
      for (int i = 0; i < PR_RL; ++i) {
        rest[i] = T(0);
        if (q0 + i * qs < w) gotr &= PrWord<T>::get(grow + q0 + i * qs, rest[i], stamp);
      }
      if (!got) {
        fetch(grow + j, piv, stamp);
        fetch(grow + w, rinv, stamp);
        if (j + 1 < w) fetch(grow + j + 1, u1, stamp);
      }
      if (!GB_IN_BOUNDS(P.status, k.hi == 0u || (k.pos >= j && k.pos < P.m))) k.pos = j;
      if (tid == 0) {
        sel = k.pos;
        if (cta == 0) {
          P.ipiv[P.kabs + j] = P.kabs + k.pos + 1;
          if (!nonzero(piv)) atomicMin(P.info, P.kabs + j + 1);
          if (is_inf_mag(pivot_mag(piv))) atomicOr(P.status, ST_RANGE);
        }
      }
      move(j, k.pos);
      if (act) {
        const T l = nonzero(piv) ? quot_rn(cur, piv, rinv) : cur;
        Sr[(size_t)j * Rs] = l;
        cur = fma(-l, u1, nxt);
        if (j + 1 < w) {
          Sr[(size_t)(j + 1) * Rs] = cur;
          best = pc_key(cur, true, pos);
        }
      }
#pragma unroll
      for (int i = 0; i < PR_RL; ++i) {
        if (q0 + i * qs < w) {
          if (!gotr) fetch(grow + q0 + i * qs, rest[i], stamp);
          pr[q0 + i * qs] = rest[i];
        }
      }
      for (int q = q0 + PR_RL * qs; q < w; q += qs) {
        T v = T(0);
        fetch(grow + q, v, stamp);
        pr[q] = v;
      }
    }
    if (j + 1 == w) break;
    ok = publish(j + 1, nbuf, best, pr);
    if (!ok) break;
    if (act) {
      const T l = Sr[(size_t)j * Rs];
      if (chain && j + 2 < w) {
        T* x = Sr + (size_t)(j + 2) * Rs;
        nxt = fma(-l, pr[j + 2], x[0]);
        x[0] = nxt;
      }
      if (upd) pc_update(Sr, Rs, pr, l, j + c_off, c_step, w);
    }
    buf = nbuf;
  }
  __threadfence();  // (after every CTA's first header: their row loads and the count's zero)
  __syncthreads();
  if (!ok || abort_flag) return;
  if (chain && live) sp[r] = GB_IN_BOUNDS(P.status, pos >= 0 && pos < P.m) ? pos : row0 + r;
  __syncthreads();
  pc_store_rows(P.A, ld, S, Rs, sp, rloc, w);
  if (chain && live && pos != row0 + r) {
    const int q = atomicAdd(P.perm, 1);
    if (GB_IN_BOUNDS(P.status, q < 2 * w)) {
      P.perm[1 + q] = pos;
      P.perm[1 + 2 * w + q] = row0 + r;
    }
  }
}

// The FP32 form: bound by the exchange, not by its pipes, so every thread polls a
// header, reads the pivot row and updates (in the roles above an 8192 x 128
// panel takes 328 us, in these 290; for FP64 it is 403 and 447)
__global__ void __launch_bounds__(PC_NTMAX, 1) panel_grid_f32_kernel(PrParams<float> P) {
  using T = float;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint4 red[PC_NTMAX / 32];   // each row group's best: key, position, row
  __shared__ uint4 red2[PC_NTMAX / 32];  // each polling warp's best: key, position, CTA
  __shared__ int abort_flag;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  const int cta = blockIdx.x, G = gridDim.x, GW = (G + 31) / 32;
  const int R = P.R, w = P.w, Rs = R | 1;
  const int64_t ld = P.ld;
  const int row0 = cta * R;
  const int rloc = max(0, min(P.m, row0 + R) - row0);
  // (row groups, classes and chain warps as in panel_cluster_kernel)
  const int RG = (R + 31) / 32;
  const int NC = nw / RG;
  const int rg = warp % RG, cls = warp / RG;
  const int r = rg * 32 + lane;
  const bool live = cls < NC && r < rloc;
  const bool chain = warp < RG;
  const size_t tile = ((size_t)w * Rs * sizeof(T) + 15) / 16 * 16;
  T* S = reinterpret_cast<T*>(smem_raw);
  T* prow = reinterpret_cast<T*>(smem_raw + tile);  // [PC_NBUF][w + 1]: pivot rows
  int* sp = reinterpret_cast<int*>(prow + (size_t)PC_NBUF * (w + 1));  // [R] positions, at the end
  T* Sr = S + r;

  if (tid == 0) {
    abort_flag = 0;
    if (cta == 0) P.perm[0] = 0;
  }
  pc_load_rows(S, Rs, P.A + (int64_t)row0 * ld, ld, rloc, w);
  __syncthreads();

  // this CTA's candidate of column c to global memory (pr as in panel_cluster_kernel)
  auto publish = [&](int c, int buf, PcKey best, const T* pr) {
    if (chain) {
      const bool own = pc_warp_best<T>(best);
      const unsigned at = __ballot_sync(0xffffffffu, own);
      if (lane == 0) red[warp] = make_uint4(best.hi, best.lo, (unsigned)best.pos, (unsigned)(rg * 32 + __ffs(at) - 1));
    }
    __syncthreads();
    uint4 e = red[lane < RG ? lane : 0];
    if (RG > 1) {
      PcKey k{lane < RG ? e.x : 0u, lane < RG ? e.y : 0u, lane < RG ? (int)e.z : INT_MAX};
      const bool own = pc_warp_best<T>(k);
      const unsigned at = __ballot_sync(0xffffffffu, own);
      e.w = __shfl_sync(0xffffffffu, e.w, at ? __ffs(at) - 1 : 0);
      e.x = k.hi;
      e.y = k.lo;
      e.z = (unsigned)k.pos;
    }
    const unsigned stamp = (unsigned)c + 1u;
    if (c == 0 && tid == nt - 1) __threadfence();  // (the CTA's row loads and the count's zero, before the barrier above)
    if (tid == nt - 1)
      pr_store(P.head + (size_t)buf * G + cta,
               make_ulonglong2(((unsigned long long)e.x << 32) | stamp,
                               ((unsigned long long)e.y << 32) | ((e.x ? e.z : 0u) << 12) | stamp));
    if (e.x != 0u) {
      auto* grow = P.rows + (size_t)(buf * G + cta) * P.rstride;
      const T* Sk = S + e.w;
      const T lc = pr != nullptr ? Sk[(size_t)(c - 1) * Rs] : T(0);
      for (int q = c + tid; q < w; q += nt) {
        T v = Sk[(size_t)q * Rs];
        if (pr != nullptr && q > c) v = fma(-lc, pr[q], v);
        PrWord<T>::put(grow + q, v, stamp);
      }
      if (warp == nw - 1) {
        const T rv = recip_rn(Sk[(size_t)c * Rs]);
        if (lane == 0) PrWord<T>::put(grow + w, rv, stamp);
      }
    }
    __syncthreads();  // (the candidate's row is read before its columns are updated)
  };
  auto fetch = [&](const typename PrWord<T>::type* q, T& v, unsigned stamp) {
    pr_fetch<T>(q, v, stamp, &abort_flag, P.status);
  };

  int pos = row0 + r;
  T cur = live ? Sr[0] : T(0);
  T nxt = live && w > 1 ? Sr[(size_t)Rs] : T(0);
  publish(0, 0, pc_key(cur, live, pos), nullptr);
  int buf = 0;
  bool ok = true;
  for (int j = 0; j < w; ++j) {
    const int nbuf = buf + 1 == PC_NBUF ? 0 : buf + 1;
    if (warp < GW) {
      PcKey k{0u, 0u, INT_MAX};
      if (tid < G) {
        const ulonglong2* hp = P.head + (size_t)buf * G + tid;
        const unsigned stamp = (unsigned)j + 1u;
        auto there = [&](const ulonglong2& h) { return (unsigned)h.x == stamp && ((unsigned)h.y & 0xfffu) == stamp; };
        ulonglong2 h = pr_load(hp);
        if (!there(h)) {
          const uint64_t t0 = gtimer();
          while (!there(h = pr_load(hp))) {
            if (*(volatile int*)&abort_flag) break;
            if (gtimer() - t0 > GB_SPIN_LIMIT_NS) {
              atomicOr(P.status, ST_TIMEOUT);
              *(volatile int*)&abort_flag = 1;
              break;
            }
          }
        }
        k.hi = (unsigned)(h.x >> 32);
        k.lo = (unsigned)(h.y >> 32);
        k.pos = k.hi ? (int)((unsigned)h.y >> 12) : INT_MAX;
      }
      __syncwarp();
      const bool own = pc_warp_best<T>(k);
      const unsigned at = __ballot_sync(0xffffffffu, own);
      if (lane == 0) red2[warp] = make_uint4(k.hi, k.lo, (unsigned)k.pos, (unsigned)(warp * 32 + (at ? __ffs(at) - 1 : 0)));
    }
    __syncthreads();
    if (abort_flag) {  // (every thread: set before this barrier, by a poll or a fetch of the column before)
      ok = false;
      break;
    }
    // the pivot, in every warp
    uint4 e = red2[lane < GW ? lane : 0];
    PcKey k{lane < GW ? e.x : 0u, lane < GW ? e.y : 0u, lane < GW ? (int)e.z : INT_MAX};
    const bool own = pc_warp_best<T>(k);
    const unsigned at = __ballot_sync(0xffffffffu, own);
    const int win = min((int)__shfl_sync(0xffffffffu, e.w, at ? __ffs(at) - 1 : 0), G - 1);
    int p = k.pos;
    if (!GB_IN_BOUNDS(P.status, k.hi == 0u || (p >= j && p < P.m))) p = j;
    const auto* grow = P.rows + (size_t)(buf * G + win) * P.rstride;
    T* pr = prow + (size_t)buf * (w + 1);
    const unsigned stamp = (unsigned)j + 1u;
    // the pivot row: what the chain needs by its warps, the rest (read after
    // the next barrier) by the others first
    T piv = T(0), rinv = T(0), u1 = T(0);
    if (chain) {
      bool got = PrWord<T>::get(grow + j, piv, stamp);
      got &= PrWord<T>::get(grow + w, rinv, stamp);
      if (j + 1 < w) got &= PrWord<T>::get(grow + j + 1, u1, stamp);
      if (!got) {
        fetch(grow + j, piv, stamp);
        fetch(grow + w, rinv, stamp);
        if (j + 1 < w) fetch(grow + j + 1, u1, stamp);
      }
    }
    for (int q = j + 1 + (tid + nt - 32 * RG) % nt; q < w; q += nt) {
      T v = T(0);
      fetch(grow + q, v, stamp);
      pr[q] = v;
    }
    if (live) {
      if (pos == p)
        pos = j;
      else if (pos == j)
        pos = p;
    }
    const bool act = live && pos > j;
    PcKey best{0u, 0u, INT_MAX};
    if (chain) {
      if (cta == 0 && tid == 0) {
        P.ipiv[P.kabs + j] = P.kabs + p + 1;
        if (!nonzero(piv)) atomicMin(P.info, P.kabs + j + 1);
        if (is_inf_mag(pivot_mag(piv))) atomicOr(P.status, ST_RANGE);
      }
      if (act) {
        const T l = nonzero(piv) ? quot_rn(cur, piv, rinv) : cur;
        Sr[(size_t)j * Rs] = l;
        cur = fma(-l, u1, nxt);
        if (j + 1 < w) {
          Sr[(size_t)(j + 1) * Rs] = cur;
          best = pc_key(cur, true, pos);
        }
      }
    }
    if (j + 1 == w) break;
    publish(j + 1, nbuf, best, pr);
    if (act) {
      const T l = Sr[(size_t)j * Rs];
      const size_t step = (size_t)NC * Rs;
      int c = j + 2 + cls;
      T* x = Sr + (size_t)c * Rs;
      if (chain && c < w) {
        nxt = fma(-l, pr[c], x[0]);
        x[0] = nxt;
        c += NC;
        x += step;
      }
      for (; c + 3 * NC < w; c += 4 * NC, x += 4 * step) {
        T v[4], u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          v[q] = x[q * step];
          u[q] = pr[c + q * NC];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q * step] = fma(-l, u[q], v[q]);
      }
      for (; c < w; c += NC, x += step) x[0] = fma(-l, pr[c], x[0]);
    }
    buf = nbuf;
  }
  __threadfence();  // (after every CTA's first header: their row loads and the count's zero)
  __syncthreads();
  if (!ok || abort_flag) return;
  if (chain && live) sp[r] = GB_IN_BOUNDS(P.status, pos >= 0 && pos < P.m) ? pos : row0 + r;
  __syncthreads();
  pc_store_rows(P.A, ld, S, Rs, sp, rloc, w);
  if (chain && live && pos != row0 + r) {
    const int q = atomicAdd(P.perm, 1);
    if (GB_IN_BOUNDS(P.status, q < 2 * w)) {
      P.perm[1 + q] = pos;
      P.perm[1 + 2 * w + q] = row0 + r;
    }
  }
}

template <typename T>
static const void* pr_kernel() {
  return sizeof(T) == 8 ? (const void*)panel_grid_f64_kernel : (const void*)panel_grid_f32_kernel;
}

// CTAs of the grid form: at least 32 rows each, at most one per SM; 0 when the
// tile does not fit.
static int pr_config(int m, int w, int tsize, const DevInfo& dev, int gmax, int* R, int* nt, size_t* smem) {
  if (w < 1 || w > 512 || m < w || gmax < 1) return 0;
  int g = dev.sm_count < gmax ? dev.sm_count : gmax;
  if (g > 32 * PR_HL) g = 32 * PR_HL;
  if ((int64_t)g * 32 > m) g = (int)cdiv(m, 32);
  *R = (int)cdiv(m, g);
  if (*R > PC_NTMAX || m >= (1 << 20)) return 0;
  *nt = *R <= (tsize == 8 ? 32 : 64) ? 256 : PC_NTMAX;
  *smem = pr_smem_bytes(*R, w, tsize);
  if (*smem + 1024 > (size_t)dev.max_smem_optin) return 0;
  return (int)cdiv(m, *R);
}

size_t panel_resident_bytes(int gmax, int wmax, int tsize) {
  return 256 + (size_t)PC_NBUF * gmax * (sizeof(ulonglong2) + (size_t)(wmax + 2) * 2 * tsize);
}

template <typename T>
int panel_resident_ctas(int m, int w, const DevInfo& dev, const PanelScratch& s) {
  int R = 0, nt = 0;
  size_t smem = 0;
  return s.xres == nullptr || w > s.wmax ? 0 : pr_config(m, w, sizeof(T), dev, s.gmax, &R, &nt, &smem);
}

template <typename T>
cudaError_t launch_panel_resident(T* Wkk, int64_t ldw, int m, int w, int kabs, int* ipiv, int* info, int* status,
                                  const PanelScratch& s, const DevInfo& dev, cudaStream_t st) {
  PrParams<T> P;
  int nt = 0;
  size_t smem = 0;
  const int G = s.xres == nullptr ? 0 : pr_config(m, w, sizeof(T), dev, s.gmax, &P.R, &nt, &smem);
  if (G <= 0 || w > s.wmax) return cudaErrorInvalidConfiguration;
  cudaError_t e = allow_max_smem(pr_kernel<T>());
  if (e != cudaSuccess) return e;
  P.A = Wkk;
  P.ld = ldw;
  P.m = m;
  P.w = w;
  P.kabs = kabs;
  P.ipiv = ipiv;
  P.info = info;
  P.status = status;
  P.perm = s.perm;
  P.head = (ulonglong2*)s.xres;
  P.rows = (typename PrWord<T>::type*)((char*)s.xres + ((size_t)PC_NBUF * s.gmax * sizeof(ulonglong2) + 127) / 128 * 128);
  P.rstride = w + 2;
  // every stamp cleared: headers and rows
  e = cudaMemsetAsync(P.head, 0, (char*)(P.rows + (size_t)PC_NBUF * G * P.rstride) - (char*)P.head, st);
  if (e != cudaSuccess) return e;
  void* args[] = {&P};
  return launch_cooperative(pr_kernel<T>(), G, nt, args, smem, st);
}

#define GB_INST(T)                                                                                            \
  template int panel_resident_ctas<T>(int, int, const DevInfo&, const PanelScratch&);                         \
  template cudaError_t launch_panel_resident<T>(T*, int64_t, int, int, int, int*, int*, int*,                 \
                                                const PanelScratch&, const DevInfo&, cudaStream_t);           \
  template bool panel_cluster_fits<T>(int, int, const DevInfo&, bool);                                              \
  template cudaError_t launch_panel_cluster<T>(T*, int64_t, int, int, int, int*, int*, int*, int*,            \
                                               const DevInfo&, cudaStream_t);
GB_INST(double)
GB_INST(float)
#undef GB_INST

}  // namespace gb
