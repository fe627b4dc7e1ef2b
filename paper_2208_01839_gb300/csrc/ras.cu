// Restricted additive Schwarz preconditioner (Eq. RAS) with block-ILU(k)
// subdomain solves, and the coarse correction of Section 3.1 with the
// per-subdomain, per-compartment constant coarse space Z:
//   z = sum_p R_p^T D_p (L_p U_p)^{-1} R_p r  +  Z A_c^{-1} Z^T r,  A_c = Z^T J Z,
// applied additively or, as in Eq. RAS_2L, multiplicatively (the J Z blocks
// summed at set-up turn the second residual update into k_az_sub).
// One CTA per subdomain for the factorization and the solves; rows of one
// level of the factors' dependency DAG are independent and run in parallel, with
// a barrier between stages.  The solve works on factors scaled by the inverted
// pivots and numbers a subdomain's solution entries by their position in the
// sweep.  The coarse matrix is block-banded
// (subdomains in reverse Cuthill-McKee order) and factored by block LU with 5x5
// pivot blocks inverted under partial pivoting, then inverted explicitly.
#include <algorithm>
#include <cmath>

#include "kernels.cuh"

namespace seird {

namespace {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ double fmaT(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fmaT(float a, float b, float c) { return fmaf(a, b, c); }

// |x| as an ordered integer key: for a value with its sign bit cleared, the
// bit pattern read as an integer grows with the magnitude (NaN above inf), so
// the pivot search runs on the integer pipe instead of GB300's narrow FP64 one.
__device__ __forceinline__ long long mag_key(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; }
__device__ __forceinline__ long long mag_key(float x) { return (long long)(__float_as_int(x) & 0x7fffffff); }
__device__ __forceinline__ bool key_ok(double, long long k) { return k != 0 && k <= 0x7ff0000000000000LL; }
__device__ __forceinline__ bool key_ok(float, long long k) { return k != 0 && k <= 0x7f800000LL; }

// Inverse of a 5x5 block by Gauss-Jordan with partial pivoting (largest |entry|
// of the column at or below the diagonal, ties to the lower row index), one
// warp: lane 5 r + c < 25 holds entry (r, c) of the block and of the identity
// it turns into the inverse, so each elimination step is two FP64 FMAs per
// lane.  Sets ERR_SINGULAR (2) on a zero (or NaN) pivot.
template <class T>
__device__ void warp_inv5(const T* __restrict__ D, T* __restrict__ out, int lane, int32_t* err) {
  const int r = lane / 5, c = lane - 5 * (lane / 5);
  const bool act = lane < 25;
  T a = act ? D[lane] : T(0);
  T b = (act && r == c) ? T(1) : T(0);
  bool sing = false;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    int piv = k;
    long long best = mag_key(__shfl_sync(FULL, a, 5 * k + k));
#pragma unroll
    for (int q = k + 1; q < 5; ++q) {
      const long long kq = mag_key(__shfl_sync(FULL, a, 5 * q + k));
      if (kq > best) {
        best = kq;
        piv = q;
      }
    }
    if (!key_ok(T(0), best)) sing = true;
    const int src = (r == k) ? 5 * piv + c : (r == piv ? 5 * k + c : lane);
    a = __shfl_sync(FULL, a, src & 31);
    b = __shfl_sync(FULL, b, src & 31);
    const T pinv = T(1) / __shfl_sync(FULL, a, 5 * k + k);
    if (r == k) {
      a *= pinv;
      b *= pinv;
    }
    const T f = __shfl_sync(FULL, a, (5 * r + k) & 31);
    const T pa = __shfl_sync(FULL, a, (5 * k + c) & 31);
    const T pb = __shfl_sync(FULL, b, (5 * k + c) & 31);
    if (act && r != k) {
      a = fmaT(-f, pa, a);
      b = fmaT(-f, pb, b);
    }
  }
  if (act) out[lane] = b;
  if (sing && lane == 0) atomicOr(err, 2);
}

template <class T>
__device__ __forceinline__ T* fvals(const RasDev& d);
template <>
__device__ __forceinline__ double* fvals<double>(const RasDev& d) { return d.fval; }
template <>
__device__ __forceinline__ float* fvals<float>(const RasDev& d) { return d.fval32; }
template <class T>
__device__ __forceinline__ T* dinvs(const RasDev& d);
template <>
__device__ __forceinline__ double* dinvs<double>(const RasDev& d) { return d.dinv; }
template <>
__device__ __forceinline__ float* dinvs<float>(const RasDev& d) { return d.dinv32; }
template <class T>
__device__ __forceinline__ T* ywk(const RasDev& d);
template <>
__device__ __forceinline__ double* ywk<double>(const RasDev& d) { return d.ywork; }
template <>
__device__ __forceinline__ float* ywk<float>(const RasDev& d) { return d.ywork32; }
template <class T>
__device__ __forceinline__ T* zwk(const RasDev& d);
template <>
__device__ __forceinline__ double* zwk<double>(const RasDev& d) { return d.zwork; }
template <>
__device__ __forceinline__ float* zwk<float>(const RasDev& d) { return d.zwork32; }

template <class T>
__device__ __forceinline__ const T* solve_fwd(const RasDev& d);
template <>
__device__ __forceinline__ const double* solve_fwd<double>(const RasDev& d) { return d.fL; }
template <>
__device__ __forceinline__ const float* solve_fwd<float>(const RasDev& d) { return d.fL32; }
template <class T>
__device__ __forceinline__ const T* solve_bwd(const RasDev& d);
template <>
__device__ __forceinline__ const double* solve_bwd<double>(const RasDev& d) { return d.bU; }
template <>
__device__ __forceinline__ const float* solve_bwd<float>(const RasDev& d) { return d.bU32; }

// Inverses of the 5x5 pivot blocks of up to six rows by one warp, in place by Gauss-Jordan
// with partial pivoting (as warp_inv5): five lanes a row, lane 5 w + c holding column c.
// An FP64 instruction holds a warp for 64 clocks whatever its lanes, so six rows at once
// cost the FP64 pipe a sixth of one row on 25 lanes.  `blk` is the row's diagonal block
// in fval, or -1; every lane of the warp calls it.
template <class T>
__device__ void rows_inv5(const T* __restrict__ fval, int64_t blk, T* __restrict__ out, int lane, int32_t* err) {
  const int w = lane / 5, c = lane - 5 * w;
  const bool act = lane < 30 && blk >= 0;
  T a[5];
#pragma unroll
  for (int r = 0; r < 5; ++r) a[r] = act ? fval[25 * blk + 5 * r + c] : (r == c ? T(1) : T(0));
  int piv[5];
  bool sing = false;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    // pivot of column k (held by lane 5 w + k): largest magnitude at or below the diagonal
    int p = k;
    long long best = mag_key(a[k]);
#pragma unroll
    for (int q = k + 1; q < 5; ++q) {
      const long long kq = mag_key(a[q]);
      if (kq > best) {
        best = kq;
        p = q;
      }
    }
    const int from = (5 * w + k) & 31;
    sing |= __shfl_sync(FULL, (int)!key_ok(T(0), best), from) != 0;
    p = __shfl_sync(FULL, p, from);
    piv[k] = p;
#pragma unroll
    for (int q = k + 1; q < 5; ++q)
      if (p == q) {
        const T t = a[k];
        a[k] = a[q];
        a[q] = t;
      }
    const T pinv = T(1) / __shfl_sync(FULL, a[k], from);
    T f[5];
#pragma unroll
    for (int r = 0; r < 5; ++r) f[r] = __shfl_sync(FULL, a[r], from);
    // column k turns into column k of the inverse so far: its unit entry starts from e_k
    if (c == k) {
#pragma unroll
      for (int r = 0; r < 5; ++r) a[r] = r == k ? T(1) : T(0);
    }
    a[k] *= pinv;
#pragma unroll
    for (int r = 0; r < 5; ++r)
      if (r != k) a[r] = fmaT(-f[r], a[k], a[r]);
  }
  // the row exchanges are column exchanges of the inverse, undone last first
  int dest = c;
#pragma unroll
  for (int k = 4; k >= 0; --k) dest = dest == k ? piv[k] : dest == piv[k] ? k : dest;
  if (act) {
#pragma unroll
    for (int r = 0; r < 5; ++r) out[5 * r + dest] = a[r];
    if (sing && c == 0) atomicOr(err, 2);
  }
}

// Block ILU(k) of R_p J R_p^T on the set-up's pattern (ILU(0): the pattern of R_p J R_p^T;
// fill blocks start at zero), IKJ form, rows in forward-level order, in the arithmetic of T
// (FP64, or FP32 for the mixed-precision path).  A warp eliminates a row whose blocks it
// holds in shared memory, lane e < 25 keeping entry e of every block (so no lane reads
// another's), with the upper blocks of earlier rows scaled by their inverted pivots:
// A_ij -= A_ik (U_kk^{-1} U_kj), so that the lower blocks stay A_ik = L_ik U_kk.  The
// level's pivot blocks are then inverted six to a warp and its upper blocks scaled.
// Bound by latency where few subdomains share the GPU (indices and the next pair's source
// block are in flight while a pair is applied) and by the FP64 pipe with many.  Rows of
// more than FACTOR_CAP blocks are eliminated in global memory.
constexpr int FACTOR_CAP = 32;

template <class T>
__device__ __forceinline__ void load_col5(const T* __restrict__ blk, int cc, bool act, T (&u)[5]) {
#pragma unroll
  for (int mm = 0; mm < 5; ++mm) u[mm] = act ? blk[5 * mm + cc] : T(0);
}

template <class T, class TV, int NT, int PER_SM>
__global__ void __launch_bounds__(NT, PER_SM) k_ilu_factor(RasDev d, const TV* __restrict__ val, int32_t* err) {
  extern __shared__ __align__(16) unsigned char fsm[];
  T* fval = fvals<T>(d);
  T* dinv = dinvs<T>(d);
  const int p = d.sd_sched[blockIdx.x];
  const int32_t r0 = d.sd_row0[p];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int rr = lane / 5, cc = lane - 5 * rr;
  const bool act = lane < 25;
  T* row = reinterpret_cast<T*>(fsm) + warp * (FACTOR_CAP * 25) + lane;  // entry `lane` of block b at row[25 b]
  const int32_t* lev = d.fwd_lev + d.sd_fwd_lev0[p];
  const int32_t nlev = d.sd_fwd_lev0[p + 1] - d.sd_fwd_lev0[p] - 1;
  // this warp's rows, level by level: lane b holds the J block of block b, lane t update pair t
  struct Next {
    int32_t lv, ri;
    int4 rec;
    int64_t u0;
    int32_t g;
    int2 pr;
  } nx;
  auto seek = [&](int32_t lv, int32_t ri) {  // first row at or after ri of level lv that is this warp's; its record
    while (lv < nlev && ri >= lev[lv + 1]) {
      ++lv;
      if (lv < nlev) ri = lev[lv] + warp;
    }
    nx.lv = lv;
    nx.ri = ri;
    if (lv < nlev) {
      nx.rec = d.frec[r0 + ri];
      nx.u0 = d.fpair[r0 + ri];
    }
  };
  auto fetch = [&] {
    if (nx.lv < nlev) {
      nx.g = lane < (nx.rec.z & 0xffff) ? d.l_gblk[nx.rec.y + lane] : -1;
      nx.pr = lane < nx.rec.w ? d.upd[nx.u0 + lane] : make_int2(0, 0);
    }
  };
  // with one CTA per SM there are registers for the next row's J blocks and pairs too
  constexpr bool AHEAD = NT == 512;
  seek(0, warp);
  if (AHEAD) fetch();
  for (int32_t lv = 0; lv < nlev; ++lv) {
    const int32_t s = lev[lv], e = lev[lv + 1];
    while (nx.lv == lv) {
      if (!AHEAD) fetch();
      const int64_t a0 = nx.rec.y, u0 = nx.u0;
      const int nb = nx.rec.z & 0xffff, npair = nx.rec.w;
      const int32_t g = nx.g;
      int2 pr = nx.pr;
      seek(lv, nx.ri + nw);
      if (nb > FACTOR_CAP) {
        for (int b = 0; b < nb; ++b) {
          const int32_t gb = d.l_gblk[a0 + b];
          if (act) fval[25 * (a0 + b) + lane] = gb >= 0 ? (T)val[25 * (int64_t)gb + lane] : T(0);
        }
        T A[5];
        for (int t = 0, j = -1; t < npair; ++t) {
          const int2 q = d.upd[u0 + t];
          if (q.x >> 16 != j) {
            j = q.x >> 16;
            const T x = act ? fval[25 * (a0 + j) + lane] : T(0);
#pragma unroll
            for (int mm = 0; mm < 5; ++mm) A[mm] = __shfl_sync(FULL, x, (5 * rr + mm) & 31);
          }
          if (act) {
            T* dst = fval + 25 * (a0 + (q.x & 0xffff)) + lane;
            T y = *dst;
#pragma unroll
            for (int mm = 0; mm < 5; ++mm) y = fmaT(A[mm], fval[25 * (int64_t)q.y + 5 * mm + cc], y);
            *dst = y;
          }
        }
        if (AHEAD) fetch();
        continue;
      }
      T U[5];
      if (npair) load_col5(fval + 25 * (int64_t)__shfl_sync(FULL, pr.y, 0), cc, act, U);
      for (int b = 0; b < nb; b += 4) {
        T v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int32_t gb = __shfl_sync(FULL, g, (b + u) & 31);
          v[u] = act && b + u < nb && gb >= 0 ? (T)val[25 * (int64_t)gb + lane] : T(0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (act && b + u < nb) row[25 * (b + u)] = v[u];
      }
      T A[5];
      int j = -1;
#pragma unroll 1
      for (int t = 0; t < npair; ++t) {  // A_ij -= A_ik (U_kk^{-1} U_kj)
        const int at = __shfl_sync(FULL, pr.x, t & 31);
        if (at >> 16 != j) {  // the next lower block: row rr of it in this lane
          j = at >> 16;
          const T x = act ? row[25 * j] : T(0);
#pragma unroll
          for (int mm = 0; mm < 5; ++mm) A[mm] = __shfl_sync(FULL, x, (5 * rr + mm) & 31);
        }
        T* dst = row + 25 * (at & 0xffff);
        T y = act ? *dst : T(0);
        T Uc[5];
#pragma unroll
        for (int mm = 0; mm < 5; ++mm) Uc[mm] = U[mm];
        if (t + 1 < npair) {  // the next pair's source block
          if (((t + 1) & 31) == 0) pr = t + 1 + lane < npair ? d.upd[u0 + t + 1 + lane] : make_int2(0, 0);
          load_col5(fval + 25 * (int64_t)__shfl_sync(FULL, pr.y, (t + 1) & 31), cc, act, U);
        }
#pragma unroll
        for (int mm = 0; mm < 5; ++mm) y = fmaT(A[mm], Uc[mm], y);
        if (act) *dst = y;
      }
      if (AHEAD) fetch();
      if (act)
        for (int b = 0; b < nb; ++b) fval[25 * (a0 + b) + lane] = row[25 * b];
    }
    __syncthreads();
    for (int32_t ri = s + 6 * warp; ri < e; ri += 6 * nw) {
      const int32_t q = ri + lane / 5;
      const int4 rec = lane < 30 && q < e ? d.frec[r0 + q] : make_int4(0, 0, 0, -1);
      rows_inv5<T>(fval, rec.w >= 0 ? (int64_t)rec.y + (rec.z >> 16) : -1, dinv + 25 * (int64_t)rec.x, lane, err);
    }
    __syncthreads();
    // upper blocks U_ij -> -U_ii^{-1} U_ij
    for (int32_t ri = s + warp; ri < e; ri += nw) {
      const int4 rec = d.frec[r0 + ri];
      T D[5];
#pragma unroll
      for (int mm = 0; mm < 5; ++mm) D[mm] = act ? dinv[25 * (int64_t)rec.x + 5 * rr + mm] : T(0);
      const int64_t end = (int64_t)rec.y + (rec.z & 0xffff);
      for (int64_t b = (int64_t)rec.y + (rec.z >> 16) + 1; b < end; b += 2) {  // two blocks in flight
        const bool two = b + 1 < end;
        T u[5], u2[5], v = T(0), v2 = T(0);
        load_col5(fval + 25 * b, cc, act, u);
        load_col5(fval + 25 * (two ? b + 1 : b), cc, act, u2);
#pragma unroll
        for (int mm = 0; mm < 5; ++mm) v = fmaT(-D[mm], u[mm], v);
        if (two) {
#pragma unroll
          for (int mm = 0; mm < 5; ++mm) v2 = fmaT(-D[mm], u2[mm], v2);
        }
        __syncwarp();  // every lane has read the blocks
        if (act) {
          fval[25 * b + lane] = v;
          if (two) fval[25 * (b + 1) + lane] = v2;
        }
      }
    }
    __syncthreads();
  }
}

// ---- subdomain solves ---------------------------------------------------------
//
// The solve reads the factors from a copy in level order (SolvePlan), scaled so that a
// row's result is one sum of block products: Dinv_i, -Dinv_i L_ij U_jj and -Dinv_i U_ij.  Every level of the
// forward (then backward) sweep is one contiguous range of padded blocks (25 values and
// the block's local column in slot 25; 26 doubles or 28 floats, so a block is a multiple
// of 16 bytes), which streams into shared memory by cp.async.bulk while earlier levels
// compute.

template <class T>
struct SolveBS;
template <>
struct SolveBS<double> {
  static constexpr int v = 26;
};
template <>
struct SolveBS<float> {
  static constexpr int v = 28;
};

__device__ __forceinline__ int col_of(double x) { return (int)__double_as_longlong(x); }
__device__ __forceinline__ int col_of(float x) { return __float_as_int(x); }
__device__ __forceinline__ void put_col(double* p, int c) { *p = __longlong_as_double((long long)c); }
__device__ __forceinline__ void put_col(float* p, int c) { *p = __int_as_float(c); }

// The solve's copy of the factors: block b is Dinv_R (src = -1 - R), or from factor block src
// of row R = brow: -Dinv_R A for a lower block (the forward plan), the block as it is for
// an upper one (backward).  One thread per value.
template <class T, bool FWD>
__global__ void __launch_bounds__(256) k_ilu_reorg(int64_t nblk, const int64_t* __restrict__ src,
                                                   const int32_t* __restrict__ col, const int32_t* __restrict__ brow,
                                                   const T* __restrict__ fval, const T* __restrict__ dinv,
                                                   T* __restrict__ out) {
  constexpr int BS = SolveBS<T>::v;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < nblk * BS;
       g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = g / BS;
    const int e = (int)(g - b * BS);
    if (e < 25) {
      const int64_t s = src[b];
      const T* D = FWD ? dinv + 25 * (int64_t)brow[b] : nullptr;
      if (!FWD) {
        out[g] = fval[25 * s + e];
      } else if (s >= 0) {
        const int r = e / 5, c = e - 5 * r;
        const T* A = fval + 25 * s + c;
        T v = T(0);
#pragma unroll
        for (int mm = 0; mm < 5; ++mm) v = fmaT(-D[5 * r + mm], A[5 * mm], v);
        out[g] = v;
      } else {
        out[g] = D[e];
      }
    } else if (e == 25) {  // window offset of the entry in bytes, or -1 - position where the plan says "far"
      const int c = col[b];
      put_col(out + g, c >= 0 ? (c & (SOLVE_WIN - 1)) * SOLVE_STRIDE<T> * (int)sizeof(T) : c);
    } else {
      out[g] = T(0);
    }
  }
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait: gives up after `polls` polls (none when polls <= 0) and reports it
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int polls) {
  for (int it = 0; it < polls; ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}
// the wait for issued copies to land before a CTA exits: never shortened, so no bulk
// copy is in flight into the shared memory of a CTA that has left
constexpr int SOLVE_DRAIN_POLLS = 1 << 20;

// Stage data of one subdomain stream through shared memory: the factor blocks, the row
// records and the rows' first values (r in the forward sweep, the forward result in the
// backward one).  Two warps bring them, up to SOLVE_SLOTS stages ahead and as far as the
// rings have room: one thread issues the bulk copies (records, blocks, the backward sweep's
// first values; "recs" and "blks" mbarriers), one warp gathers a forward stage's r by
// cp.async once its records are here ("vals").  Where a stage goes and which stage must have
// been consumed before it is part of the stage's record, so each of the two has one wait a
// stage; the blocks are also drawn into L2 ahead of their copies.  The consumer warps take
// the stages in order and meet at a named barrier after each one (the rows of a level depend
// on the rows of earlier levels), which the last of them joins when the next stage has
// arrived, so that the others have no wait of their own; a stage's "empty" mbarrier then
// completes.  (A test of a completed mbarrier takes 46 clocks, a barrier of eight warps
// 28.)  Every wait is bounded; on a timeout the
// kernel sets bit 3 of *err, lets every issued copy land and returns.
// The work arrays y and z hold one padded row per sweep position.  The forward sweep leaves
// its results in y, and in z at the row's backward position, where the backward sweep finds
// its first values as one contiguous run a stage and leaves its results.  The last SOLVE_WIN
// results of a sweep also stay in shared memory, where nearly all of a row's dependencies
// lie; which ones do not is known at set-up (HostSetup::SolvePlan::col).
// Ring of factor blocks: several stages, or one (118 blocks), which leaves the shared memory
// to more resident subdomains (solve_ring_blocks).  How far the copies run ahead is what
// bounds a stage once its own chain is short: 128 subdomains of 4400 rows, ILU(1), take 1.74
// ms in FP64 (1.20 in FP32) with the short ring and 1.12 (0.61) with the long one.
// Measured for a preconditioner apply without a coarse space (one sweep pair and the two
// index permutations), start of these sweeps -> now: 1024 x 1024 nodes, 512 subdomains, ILU(1)
// 1.24 -> 1.04 ms FP64, 0.69 -> 0.50 ms FP32; 501k nodes, 128 subdomains, ILU(1) 1.67 -> 1.12
// and 0.97 -> 0.61 ms; 16 subdomains of 4489 rows, ILU(0) 0.94 -> 0.76 and 0.57 -> 0.45 ms.
constexpr int SOLVE_AHEAD = 320;  // blocks drawn into L2 ahead of their copies

__device__ __forceinline__ void mbar_init_count(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// one arrival on `bar` when every cp.async this thread has issued so far has landed (the
// arrival is part of the barrier's count)
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// five values of r: doubles at stride 5, or floats padded to stride 8
__device__ __forceinline__ void cp_async_row(double* dst, const double* r, int64_t i) {
  const uint32_t d = smem_u32(dst);
#pragma unroll
  for (int c = 0; c < 5; ++c)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d + 8 * c), "l"(r + 5 * i + c) : "memory");
}
__device__ __forceinline__ void cp_async_row(float* dst, const float* r, int64_t i) {
  const uint32_t d = smem_u32(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(r + 8 * i) : "memory");
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 16), "l"(r + 8 * i + 4) : "memory");
}
// this thread's stores before it are seen by bulk copies issued after a synchronisation
// that follows it
__device__ __forceinline__ void fence_bulk() { asm volatile("fence.proxy.async;" ::: "memory"); }
// named barrier 1 over the NC consumer warps
template <int NC>
__device__ __forceinline__ void consumers_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * NC) : "memory");
}

// five values of a row of a work array or of the window (16-byte aligned)
__device__ __forceinline__ void load5(const double* p, double (&v)[5]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x;
  v[1] = a.y;
  v[2] = b.x;
  v[3] = b.y;
  v[4] = p[4];
}
__device__ __forceinline__ void load5(const float* p, float (&v)[5]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  v[0] = a.x;
  v[1] = a.y;
  v[2] = a.z;
  v[3] = a.w;
  v[4] = p[4];
}

// Consumer warps of the two CTA shapes: 7 names the one of 256 threads (six consumers and the
// two copying warps), 3 the one of 160 (three and two).  Every row's arithmetic is the same.
constexpr int solve_consumers(int ncw) { return ncw == 7 ? 6 : 3; }

template <class T, class TZ, int NCW, int RB, bool WIDE>
__global__ void __launch_bounds__(32 * (solve_consumers(NCW) + 2), NCW <= 3 ? 6 : 4)
    k_ilu_solve(RasDev d, const T* __restrict__ r, TZ* __restrict__ z, int32_t* err) {
  constexpr int NC = solve_consumers(NCW);
  constexpr int BS = SolveBS<T>::v, BSB = BS * (int)sizeof(T);
  constexpr int RR = solve_ring_rows(RB);
  constexpr int RBP = RB + SOLVE_RING_SPARE, RV = RB == SOLVE_RING_HALF ? 1 : 0;
  constexpr int NS = SOLVE_SLOTS;
  constexpr int W = SOLVE_STRIDE<T>, WB = W * (int)sizeof(T);
  extern __shared__ __align__(128) unsigned char smem[];  // factor ring, first values, window
  constexpr int FV = RBP * BSB, WIN = FV + RR * WB;
  __shared__ __align__(8) uint64_t recs[NS], blks[NS], vals[NS], empty[NS];
  __shared__ __align__(16) int4 info[RR];
  __shared__ __align__(16) int4 slot[NS];  // byte offset of the blocks, first row of the row rings, rows (| 256: `ahead`), first position
  __shared__ int abort_at;  // first stage at which a consumer warp's wait gave up (INT_MAX: none)
  const int p = d.sd_sched[blockIdx.x];
  const int32_t r0 = d.sd_row0[p];
  T* const y = ywk<T>(d) + (int64_t)W * r0;
  T* const zz = zwk<T>(d) + (int64_t)W * r0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int32_t LF = d.fwd.sd_lev0[p], nF = d.fwd.sd_lev0[p + 1] - LF - 1;
  const int32_t LB = d.bwd.sd_lev0[p], nB = d.bwd.sd_lev0[p + 1] - LB - 1;
  const int nstage = nF + nB;
  if (tid == 0) {
    for (int k = 0; k < NS; ++k) {
      mbar_init_count(&recs[k], 1);
      mbar_init_count(&blks[k], 1);
      mbar_init_count(&vals[k], 32);
      mbar_init_count(&empty[k], 1);
    }
    abort_at = INT_MAX;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // stage g < nF is forward level g, otherwise backward level g - nF; it uses slot g % NS,
  // whose barriers complete phase (g / NS) & 1 for it (forward stages come first, so this
  // holds for the gathered ones too)
  auto phase = [](int g) { return (uint32_t)((g / NS) & 1); };

  if (warp == NC) {
    // ---- bulk copies (one thread); stage records are read four stages ahead
    if (lane != 0) return;
    auto record = [&](int g) {
      if (g >= nstage) return make_int4(0, 0, 0, 0);
      return g < nF ? d.fwd.stage[LF + g] : d.bwd.stage[LB + g - nF];
    };
    int4 st[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) st[u] = record(u);
    int pf = st[0].y, pend = 0;  // L2 prefetch: next block, end of the sweep's blocks
    int gi = 0;
    bool ok = true;
    while (ok && gi < nstage) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (ok && gi < nstage) {
          const int4 s = st[u];
          st[u] = record(gi + 4);
          const bool fw = gi < nF;
          const int sl = gi % NS, nr = stage_rows(s), nb = stage_blocks(s);
          const int dist = stage_distance(s, RV);
          if (dist != SOLVE_FREE) ok = mbar_wait(&empty[(gi - dist) % NS], phase(gi - dist), d.wait_polls);
          if (ok) {
            const int rb = stage_block_offset(s, RV), rr = stage_row_offset(s, RV);
            const bool ahead = stage_distance(st[(u + 1) & 3], RV) >= 2;  // the next stage does not wait for this one
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            slot[sl] = make_int4(rb * BSB, rr, nr | (int)ahead << 8, s.x);
            const uint32_t bytes_b = (uint32_t)nb * BSB, bytes_i = (uint32_t)nr * (uint32_t)sizeof(int4);
            const uint32_t bytes_v = fw ? 0u : (uint32_t)nr * WB;
            const T* F = fw ? solve_fwd<T>(d) : solve_bwd<T>(d);
            mbar_arrive_tx(&recs[sl], bytes_i);  // releases the slot with the records
            if (bytes_i) bulk_g2s(info + rr, (fw ? d.fwd : d.bwd).info + r0 + s.x, bytes_i, &recs[sl]);
            mbar_arrive_tx(&blks[sl], bytes_b + bytes_v);
            if (bytes_b) bulk_g2s(smem + rb * BSB, F + (int64_t)s.y * BS, bytes_b, &blks[sl]);
            if (bytes_v) bulk_g2s(smem + FV + rr * WB, zz + (int64_t)W * s.x, bytes_v, &blks[sl]);
            if (gi == 0 || gi == nF) {
              pf = s.y + nb;
              const int4 last = fw ? d.fwd.stage[LF + nF - 1] : d.bwd.stage[LB + nB - 1];
              pend = last.y + stage_blocks(last);
            }
            while (pf < pend && pf < s.y + SOLVE_AHEAD) {
              const int n = min(64, pend - pf);
              asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(F + (int64_t)pf * BS), "r"((uint32_t)n * BSB)
                           : "memory");
              pf += n;
            }
            ++gi;
          }
        }
      }
    }
    if (!ok) atomicOr(err, 8);
    // every issued copy lands before the CTA can exit (the last stage issued on
    // each slot is the only one whose phases may still be open)
    for (int k = max(0, gi - NS); k < gi; ++k) {
      mbar_wait(&recs[k % NS], phase(k), SOLVE_DRAIN_POLLS);
      mbar_wait(&blks[k % NS], phase(k), SOLVE_DRAIN_POLLS);
    }
    return;
  }

  if (warp == NC + 1) {
    // ---- gathers of the forward stages' r
    bool ok = true;
    for (int g = 0; g < nF && ok; ++g) {
      const int sl = g % NS;
      ok = __all_sync(FULL, mbar_wait(&recs[sl], phase(g), d.wait_polls));
      if (ok) {
        const int4 ds = slot[sl];
        for (int q = lane; q < (ds.z & 255); q += 32)
          cp_async_row(reinterpret_cast<T*>(smem + FV) + W * (ds.y + q), r, info[ds.y + q].x);
        cp_async_arrive(&vals[sl]);
      }
    }
    if (!ok && lane == 0) atomicOr(err, 8);
    asm volatile("cp.async.wait_all;" ::: "memory");
    return;
  }

  // ---- consumers (warps 0 .. NC - 1).  S lane groups to a row: a warp takes 6 / S rows,
  // lane = 5 (part (6 / S) + row) + component, and part p of a row sums its blocks p,
  // p + S, ...; the inverted pivot (forward) or the first value (backward) opens part 0.
  // An FP64 FMA holds a warp for 64 clocks whatever its lanes and dependences, and four
  // such warps fill an SM's FP64 pipe; in FP32 a stage costs its chain of instructions.
  // Both want a stage's rows spread over the warps there are, and short code.  S = 1
  // keeps the sums of a row's even and odd blocks apart and adds them at the end, as the
  // two parts of S = 2 do: the same sums in the same order, so a launch shape may take
  // either.
  const int l5 = lane / 5, cpt = lane - 5 * l5;
  auto rows = [&]<int S>(const int4 ds, int nr, bool fw, int q0) {
    constexpr int R = 6 / S;
    const int part = S == 1 ? 0 : l5 / R, q = q0 + l5 - part * R;
    const bool act = lane < 30 && q < nr;
    int4 rec = make_int4(0, 0, 0, -1);
    T acc = T(0), acc2 = T(0);
    if (act) rec = info[ds.y + q];
    const unsigned char* B = smem + ds.x + rec.y * BSB;  // the row's blocks
    const T* vec = fw ? y : zz;
    int j = part;
    if (act && part == 0) {
      const T* f = reinterpret_cast<const T*>(smem + FV) + W * (ds.y + q);
      if (fw) {
        T x[5];
        load5(f, x);
#pragma unroll
        for (int mm = 0; mm < 5; ++mm)
          if (S == 1) acc2 = fmaT(reinterpret_cast<const T*>(B)[5 * cpt + mm], x[mm], acc2);
          else acc = fmaT(reinterpret_cast<const T*>(B)[5 * cpt + mm], x[mm], acc);
        j = S;  // block 0 is done (S = 1: in the even chain, and block 1 is odd)
      } else {
        acc = f[cpt];
      }
    }
#pragma unroll 1
    for (; j < rec.z; j += S) {
      const unsigned char* Bj = B + j * BSB;
      const int c = col_of(*reinterpret_cast<const T*>(Bj + 25 * (int)sizeof(T)));
      T x[5];
      if (c >= 0) load5(reinterpret_cast<const T*>(smem + WIN + c), x);
      else load5(vec + W * ~c, x);
#pragma unroll
      for (int mm = 0; mm < 5; ++mm) acc = fmaT(reinterpret_cast<const T*>(Bj)[5 * cpt + mm], x[mm], acc);
      if (S == 1) {  // the next block belongs to the other chain
        const T t = acc;
        acc = acc2;
        acc2 = t;
      }
    }
    if (S == 1) {
      acc += acc2;  // FP addition commutes: whichever register holds which chain
    } else {
      T oth[S];
#pragma unroll
      for (int k = 1; k < S; ++k) oth[k] = __shfl_sync(FULL, acc, (lane + 5 * R * k) & 31);
      if (S == 2) acc += oth[1];
      else if (S == 3) acc += oth[1] + oth[2];
      else if (S == 6) acc = (acc + oth[S - 1]) + ((oth[1] + oth[S / 3]) + (oth[S / 2] + oth[S - 2]));
    }
    if (act && part == 0) {
      const int k = ds.w + q;
      reinterpret_cast<T*>(smem + WIN)[W * (k & (SOLVE_WIN - 1)) + cpt] = acc;
      if (fw) {
        y[W * k + cpt] = acc;
        zz[W * rec.w + cpt] = acc;
      } else {
        zz[W * k + cpt] = acc;
        if (rec.w >= 0) z[5 * (int64_t)rec.w + cpt] = (TZ)acc;
      }
    }
  };
  // One or two parts to a row give the same sums: two while a warp is left for each group
  // of three rows, else six rows to a warp with the last one to three again in two parts.
  // In FP32, where the FMAs are free, and for WIDE (no more subdomains than SMs, so that
  // nothing else uses an SM's FP64 pipe while a stage waits for its longest row): more
  // parts for the smallest stages, by their size alone.
  // A warp whose wait gives up notes the stage and takes no rows of it; all warps leave
  // after the barrier that closes that stage.
  auto arrived = [&](int g) {
    bool ok = mbar_wait(&blks[g % NS], phase(g), d.wait_polls);
    ok = ok && mbar_wait(g < nF ? &vals[g % NS] : &recs[g % NS], phase(g), d.wait_polls);
    return __all_sync(FULL, ok) != 0;
  };
  bool landed = arrived(0);
  if (!landed && lane == 0) atomicMin(&abort_at, 0);
  int g = 0;
  for (; g < nstage; ++g) {
    const int sl = g % NS;
    const int4 ds = slot[sl];
    if (*(volatile int*)&abort_at < g) break;
    const bool fw = g < nF;
    const int nr = landed ? ds.z & 255 : 0;
    if ((WIDE || sizeof(T) == 4) && nr <= 4) {
#pragma unroll 1
      for (int q = warp; q < nr; q += NC) rows.template operator()<6>(ds, nr, fw, q);
    } else if ((WIDE && nr <= 10) || (sizeof(T) == 4 && nr <= 12)) {
#pragma unroll 1
      for (int q = 2 * warp; q < nr; q += 2 * NC) rows.template operator()<3>(ds, nr, fw, q);
    } else if (nr <= 3 * NC) {
      if (3 * warp < nr) rows.template operator()<2>(ds, nr, fw, 3 * warp);
    } else {
      const int rem = nr % 6, six = rem > 3 ? nr : nr - rem;
      int q = 6 * warp;
#pragma unroll 1
      for (; q < six; q += 6 * NC) rows.template operator()<1>(ds, nr, fw, q);
      if (q == six && six < nr) rows.template operator()<2>(ds, nr, fw, q);
    }
    const bool ahead = landed && (ds.z & 256) != 0 && g + 1 < nstage;  // the next stage does not wait for this one
    if (ahead && warp == NC - 1 && !arrived(g + 1) && lane == 0) atomicMin(&abort_at, g);
    if (g == nF - 1) fence_bulk();  // the backward sweep's first values are read by bulk copies
    consumers_sync<NC>();  // every row of this stage is written; its ring space is free
    if (landed && tid == 0) mbar_arrive(&empty[sl]);
    if (!ahead && g + 1 < nstage) {
      landed = arrived(g + 1);
      if (!landed && lane == 0) atomicMin(&abort_at, g + 1);
    }
  }
  if (tid == 0 && (g < nstage || *(volatile int*)&abort_at != INT_MAX)) atomicOr(err, 8);
}

// ---- coarse space --------------------------------------------------------

// one warp per chunk of J blocks that belong to the same coarse block
template <class TV>
__global__ void k_coarse_chunks(int32_t nchunk, const int32_t* __restrict__ cptr, const int32_t* __restrict__ blk,
                                const TV* __restrict__ val, double* __restrict__ cpart) {
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (gw >= nchunk || lane >= 25) return;
  double s = 0.0;
  for (int32_t b = cptr[gw]; b < cptr[gw + 1]; ++b) s += (double)val[25 * (int64_t)blk[b] + lane];
  cpart[25 * gw + lane] = s;
}

__global__ void k_coarse_dst(int32_t ndst, const int32_t* __restrict__ dptr, const int64_t* __restrict__ didx,
                             const double* __restrict__ cpart, double* __restrict__ band) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= 25 * (int64_t)ndst) return;
  const int64_t dd = g / 25;
  const int e = (int)(g - 25 * dd);
  double s = 0.0;
  for (int32_t c = dptr[dd]; c < dptr[dd + 1]; ++c) s += cpart[25 * (int64_t)c + e];
  band[25 * didx[dd] + e] = s;
}

__device__ __forceinline__ double* bblk(double* band, int bw, int ib, int jb) {
  return band + 25 * ((int64_t)ib * (2 * bw + 1) + (jb - ib + bw));
}

// Block step kb of the banded LU, one CTA per row i in (kb, kb + bw] (one in all at the end):
// every CTA inverts the pivot block for itself (the step's latency either way), forms
// L_i,kb and updates its row, A_ij -= L_i,kb A_kb,j for j in (kb, kb + bw]; no CTA writes
// what another reads, so a step is one launch.  512 units: with a launch for the pivot column
// and one for the update 8.5 us a step at 2.0M nodes and 9.2 us at 1024 x 1024 (wider band),
// 6.7 and 7.2 us now; the pivot's serial inverse is most of it.
__global__ void __launch_bounds__(256) k_band_step(int P, int bw, int kb, double* band, double* cdinv, int32_t* err) {
  __shared__ double Dk[25], L[25];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nb = min(bw, P - 1 - kb), ib = kb + 1 + blockIdx.x;
  if (warp == 0) {
    const double a = lane < 25 && nb > 0 ? bblk(band, bw, ib, kb)[lane] : 0.0;
    warp_inv5<double>(bblk(band, bw, kb, kb), Dk, lane, err);
    __syncwarp();
    if (blockIdx.x == 0 && lane < 25) cdinv[25 * (int64_t)kb + lane] = Dk[lane];
    if (nb > 0) {
      const int rr = lane / 5, cc = lane - 5 * rr;
      double v = 0.0;
#pragma unroll
      for (int mm = 0; mm < 5; ++mm) {
        const double am = __shfl_sync(FULL, a, (5 * rr + mm) & 31);
        if (lane < 25) v = fma(am, Dk[5 * mm + cc], v);
      }
      if (lane < 25) {
        L[lane] = v;
        bblk(band, bw, ib, kb)[lane] = v;
      }
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 25 * nb; t += blockDim.x) {
    const int jb = kb + 1 + t / 25, e = t % 25, rr = e / 5, cc = e - 5 * rr;
    const double* Ak = bblk(band, bw, kb, jb);
    double v = 0.0;
#pragma unroll
    for (int mm = 0; mm < 5; ++mm) v = fma(L[5 * rr + mm], Ak[5 * mm + cc], v);
    bblk(band, bw, ib, jb)[e] -= v;
  }
}

// y <- A_c^{-1} y with the banded block LU factors (one CTA, y in shared memory).
// With unit != 0, CTA b solves for the unit vector e_b and writes row b of
// A_c^{-T} (= column b of A_c^{-1}) to yg + b*5P: the explicit inverse.
__global__ void k_band_solve(int P, int bw, const double* __restrict__ band, const double* __restrict__ cdinv,
                             double* __restrict__ yg, int unit) {
  extern __shared__ double ys[];
  const int tid = threadIdx.x, bd = blockDim.x;
  double* bandm = const_cast<double*>(band);
  if (unit) {
    for (int k = tid; k < 5 * P; k += bd) ys[k] = (k == (int)blockIdx.x) ? 1.0 : 0.0;
    yg += (int64_t)blockIdx.x * 5 * P;
  } else {
    for (int k = tid; k < 5 * P; k += bd) ys[k] = yg[k];
  }
  __syncthreads();
  for (int kb = unit ? (int)blockIdx.x / 5 : 0; kb < P; ++kb) {  // e_b is zero above block b/5
    const int nb = min(bw, P - 1 - kb);
    for (int t = tid; t < 5 * nb; t += bd) {
      const int ib = kb + 1 + t / 5, r = t % 5;
      const double* L = bblk(bandm, bw, ib, kb) + 5 * r;
      double v = 0.0;
#pragma unroll
      for (int mm = 0; mm < 5; ++mm) v = fma(L[mm], ys[5 * kb + mm], v);
      ys[5 * ib + r] -= v;
    }
    __syncthreads();
  }
  for (int kb = P - 1; kb >= 0; --kb) {
    double tmp = 0.0;
    if (tid < 5) {
      const double* Dk = cdinv + 25 * (int64_t)kb + 5 * tid;
#pragma unroll
      for (int mm = 0; mm < 5; ++mm) tmp = fma(Dk[mm], ys[5 * kb + mm], tmp);
    }
    __syncthreads();
    if (tid < 5) ys[5 * kb + tid] = tmp;
    __syncthreads();
    const int nb = min(bw, kb);
    for (int t = tid; t < 5 * nb; t += bd) {
      const int ib = kb - 1 - t / 5, r = t % 5;
      const double* Ub = bblk(bandm, bw, ib, kb) + 5 * r;
      double v = 0.0;
#pragma unroll
      for (int mm = 0; mm < 5; ++mm) v = fma(Ub[mm], ys[5 * kb + mm], v);
      ys[5 * ib + r] -= v;
    }
    __syncthreads();
  }
  for (int k = tid; k < 5 * P; k += bd) yg[k] = ys[k];
}

// Explicit inverse, one CTA per block column b of the identity: L U X = E_b for
// its five columns at once (ys[row][c] in shared memory), so a step over one
// block row of the band is 25 independent dot products per band block.  X goes
// to rows 5b..5b+4 of AinvT (row j of AinvT = column j of A_c^{-1}).  Bound by the FP64 pipe
// (five FMAs a product sum) and by the latency of a step's band blocks, which are
// therefore loaded a step ahead, INV_ITEMS sums a thread (512 units, 2.0M nodes: 4.73 -> 3.94
// ms; 1024 x 1024: 5.37 -> 4.52).
constexpr int INV_ITEMS = 3;
__global__ void __launch_bounds__(256) k_band_inv(int P, int bw, const double* __restrict__ band,
                                                  const double* __restrict__ cdinv, double* __restrict__ ainvT) {
  extern __shared__ double ys[];
  const int tid = threadIdx.x, bd = blockDim.x;
  const int b = blockIdx.x;
  double* bandm = const_cast<double*>(band);
  for (int k = tid; k < 25 * P; k += bd) ys[k] = (k / 5 == 5 * b + k % 5) ? 1.0 : 0.0;
  // item t of step kb: row r of the band block t / 25 rows below (above) kb, column cc
  auto rowp = [&](int kb, int t, bool fwd) {
    return bblk(bandm, bw, fwd ? kb + 1 + t / 25 : kb - 1 - t / 25, kb) + 5 * ((t / 5) % 5);
  };
  double A[INV_ITEMS][5];
  auto fetch = [&](int kb, bool fwd) {
    const int n = 25 * (fwd ? min(bw, P - 1 - kb) : min(bw, kb));
#pragma unroll
    for (int u = 0; u < INV_ITEMS; ++u) {
      const int t = tid + 256 * u;
      if (t < n) {
        const double* p = rowp(kb, t, fwd);
#pragma unroll
        for (int mm = 0; mm < 5; ++mm) A[u][mm] = __ldg(p + mm);
      }
    }
  };
  auto item = [&](int kb, int t, bool fwd, const double* a) {
    const int ib = fwd ? kb + 1 + t / 25 : kb - 1 - t / 25, r = (t / 5) % 5, cc = t % 5;
    double v = ys[5 * (5 * ib + r) + cc];
#pragma unroll
    for (int mm = 0; mm < 5; ++mm) v = fma(-a[mm], ys[5 * (5 * kb + mm) + cc], v);
    ys[5 * (5 * ib + r) + cc] = v;
  };
  auto step = [&](int kb, bool fwd, int next) {
    const int n = 25 * (fwd ? min(bw, P - 1 - kb) : min(bw, kb));
#pragma unroll
    for (int u = 0; u < INV_ITEMS; ++u)
      if (tid + 256 * u < n) item(kb, tid + 256 * u, fwd, A[u]);
    for (int t = tid + 256 * INV_ITEMS; t < n; t += 256) item(kb, t, fwd, rowp(kb, t, fwd));
    if (next >= 0 && next < P) fetch(next, fwd);
    __syncthreads();
  };
  fetch(b, true);
  __syncthreads();
  for (int kb = b; kb < P; ++kb) step(kb, true, kb + 1);  // E_b is zero above block row b
  fetch(P - 1, false);
  double D[5];
  auto pivot = [&](int kb) {
    if (tid < 25) {
#pragma unroll
      for (int mm = 0; mm < 5; ++mm) D[mm] = __ldg(cdinv + 25 * (int64_t)kb + 5 * (tid / 5) + mm);
    }
  };
  pivot(P - 1);
  for (int kb = P - 1; kb >= 0; --kb) {
    if (tid < 32) {  // one warp: its lanes read the five rows before they write them
      double tmp = 0.0;
      if (tid < 25) {
#pragma unroll
        for (int mm = 0; mm < 5; ++mm) tmp = fma(D[mm], ys[5 * (5 * kb + mm) + tid % 5], tmp);
      }
      __syncwarp();
      if (tid < 25) ys[5 * (5 * kb + tid / 5) + tid % 5] = tmp;
    }
    if (kb > 0) pivot(kb - 1);
    __syncthreads();
    step(kb, false, kb - 1);
  }
  const int64_t nc = 5 * (int64_t)P;
  for (int k = tid; k < 25 * P; k += bd) ainvT[(5 * b + k % 5) * nc + k / 5] = ys[k];
}

// part[chunk][i] = sum_{j in chunk} AinvT[j][i] rc[j]  (AinvT row j = column j of A_c^{-1})
constexpr int GEMV_CHUNK = 64;
__global__ void k_coarse_gemv_part(int nc, const double* __restrict__ AinvT, const double* __restrict__ rc,
                                   double* __restrict__ part) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j0 = blockIdx.y * GEMV_CHUNK;
  const int j1 = min(nc, j0 + GEMV_CHUNK);
  if (i >= nc) return;
  double s = 0.0;
  for (int j = j0; j < j1; ++j) s = fma(AinvT[(int64_t)j * nc + i], rc[j], s);
  part[(int64_t)blockIdx.y * nc + i] = s;
}

__global__ void k_coarse_gemv_sum(int nc, int nchunk, const double* __restrict__ part, double* __restrict__ y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nc) return;
  double s = 0.0;
  for (int q = 0; q < nchunk; ++q) s += part[(int64_t)q * nc + i];
  y[i] = s;
}

// crhs[cpos[p]] = Z^T r : sums of r over the nodes owned by p, per compartment
__global__ void __launch_bounds__(256) k_coarse_restrict(const int32_t* __restrict__ own_ptr,
                                                         const int32_t* __restrict__ cpos,
                                                         const double* __restrict__ r, double* __restrict__ crhs) {
  __shared__ double sh[5][8];
  const int p = blockIdx.x;
  double acc[5] = {0, 0, 0, 0, 0};
  for (int32_t i = own_ptr[p] + threadIdx.x; i < own_ptr[p + 1]; i += blockDim.x)
#pragma unroll
    for (int c = 0; c < 5; ++c) acc[c] += r[5 * (int64_t)i + c];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    double v = acc[c];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
    if ((threadIdx.x & 31) == 0) sh[c][threadIdx.x >> 5] = v;
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    double v = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += sh[threadIdx.x][w];
    crhs[5 * (int64_t)cpos[p] + threadIdx.x] = v;
  }
}

// z += Z y : every node adds its subdomain's coarse value
template <class TZ>
__global__ void k_coarse_prolong_add(int64_t n, const int32_t* __restrict__ owner, const int32_t* __restrict__ cpos,
                                     const double* __restrict__ y, TZ* __restrict__ z) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < 5 * n; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = g / 5;
    z[g] = (TZ)((double)z[g] + y[5 * (int64_t)cpos[owner[i]] + (g - 5 * i)]);
  }
}

// z += Z y in FP32 (mixed path): every node adds its unit's coarse value
__global__ void k_coarse_prolong_add32(int64_t n, const int32_t* __restrict__ owner, const int32_t* __restrict__ cpos,
                                       const float* __restrict__ y, float* __restrict__ z) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < 5 * n; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = g / 5;
    z[g] += y[5 * (int64_t)cpos[owner[i]] + (g - 5 * i)];
  }
}

__global__ void k_coarse_to_f32(int n, const double* __restrict__ y, float* __restrict__ y32) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < n) y32[g] = (float)y[g];
}

}  // namespace

// 16 warps a CTA while every CTA has an SM to itself (a level's rows are then all in flight), 8
// with more; in FP64 three such CTAs per SM, whose registers hold the kernel, up to four
// subdomains per SM, and four beyond (1024 x 1024 nodes, FP64, three against four: 256
// subdomains, ILU(0) 9.8 against 11.5 ms a set-up, 512, ILU(1) 11.4 against 11.6, 2048, ILU(3)
// 35.4 against 33.5).  Set-ups at the start of this form -> now: 501k nodes, 128 subdomains,
// ILU(1) 15.9 -> 7.6 ms FP64, 10.8 -> 3.8 ms FP32; 1024 x 1024, 512 subdomains, ILU(1) 15.4 ->
// 11.4 and 8.0 -> 5.4 ms; 16 subdomains of 4489 rows, ILU(0) 11.2 -> 4.6 and 6.8 -> 2.1 ms.
template <class T, class TV>
void launch_ilu_factor_t(const RasDev& d, const TV* val, int32_t* err, cudaStream_t s) {
  constexpr size_t row = FACTOR_CAP * 25 * sizeof(T);
  constexpr int few = sizeof(T) == 8 ? 3 : 4;
  if (d.P <= SOLVE_WIDE_MAX) k_ilu_factor<T, TV, 512, 1><<<d.P, 512, 16 * row, s>>>(d, val, err);
  else if (d.P <= 4 * SOLVE_WIDE_MAX) k_ilu_factor<T, TV, 256, few><<<d.P, 256, 8 * row, s>>>(d, val, err);
  else k_ilu_factor<T, TV, 256, 4><<<d.P, 256, 8 * row, s>>>(d, val, err);
}
void launch_ilu_factor(const RasDev& d, const double* val, const float* val32, int32_t* err, bool fp32,
                       cudaStream_t s) {
  if (fp32) launch_ilu_factor_t<float>(d, val32, err, s);
  else launch_ilu_factor_t<double>(d, val, err, s);
  count_launch();
}

// dynamic shared memory of a solve CTA: factor ring, first values, window of results
template <class T>
constexpr size_t solve_smem(int ring_blocks) {
  return ((size_t)(ring_blocks + SOLVE_RING_SPARE) * SolveBS<T>::v + SOLVE_STRIDE<T> * (solve_ring_rows(ring_blocks) + SOLVE_WIN)) *
         sizeof(T);
}

void launch_ilu_reorg(const RasDev& d, int64_t nfwd, int64_t nbwd, const int64_t* fsrc, const int32_t* fcol,
                      const int32_t* frow, const int64_t* bsrc, const int32_t* bcol, bool fp32, cudaStream_t s) {
  const int grid = 152 * 8;
  if (fp32) {
    k_ilu_reorg<float, true><<<grid, 256, 0, s>>>(nfwd, fsrc, fcol, frow, d.fval32, d.dinv32, d.fL32);
    k_ilu_reorg<float, false><<<grid, 256, 0, s>>>(nbwd, bsrc, bcol, nullptr, d.fval32, d.dinv32, d.bU32);
  } else {
    k_ilu_reorg<double, true><<<grid, 256, 0, s>>>(nfwd, fsrc, fcol, frow, d.fval, d.dinv, d.fL);
    k_ilu_reorg<double, false><<<grid, 256, 0, s>>>(nbwd, bsrc, bcol, nullptr, d.fval, d.dinv, d.bU);
  }
  count_launch();
  count_launch();
}

// f.template operator()<NCW, RB, WIDE>() for the launch shape of d
template <class T, class F>
void solve_variant(const RasDev& d, F&& f) {
  auto warps = [&]<int RB, bool WIDE>() {
    if (d.solve_warps == 3) f.template operator()<3, RB, WIDE>();
    else f.template operator()<7, RB, WIDE>();
  };
  auto ring = [&]<int A, int B, int C>() {
    if (d.solve_ring == SOLVE_RING_HALF) warps.template operator()<SOLVE_RING_HALF, false>();
    else if (d.solve_ring == A) warps.template operator()<A, false>();
    else if (d.solve_ring == B) warps.template operator()<B, false>();
    else warps.template operator()<C, false>();
  };
  if (d.P <= SOLVE_WIDE_MAX) {
    if (d.solve_ring == SOLVE_RING_HALF) warps.template operator()<SOLVE_RING_HALF, true>();
    else warps.template operator()<SOLVE_RING_1, true>();
  } else if constexpr (sizeof(T) == 8) {
    ring.template operator()<SOLVE_RING_2, SOLVE_RING_3, SOLVE_RING_4>();
  } else {
    ring.template operator()<SOLVE_RING_2, SOLVE_RING_4F, SOLVE_RING_FULL>();
  }
}

// CTAs take the subdomains longest first (sd_sched): with several waves the short ones fill
// the tail (18.4M nodes, 4096 subdomains: 7.5% off the solve), in one wave it decides which
// share an SM (1024 x 1024, 512 subdomains: 1.07 -> 1.03 ms in FP64, 0.532 -> 0.525 in FP32).
template <class T>
void launch_ilu_solve_t(const RasDev& d, const T* r, T* z, int32_t* err, cudaStream_t s) {
  solve_variant<T>(d, [&]<int NCW, int RB, bool WIDE>() {
    k_ilu_solve<T, T, NCW, RB, WIDE><<<d.P, 32 * (solve_consumers(NCW) + 2), solve_smem<T>(RB), s>>>(d, r, z, err);
  });
  count_launch();
}

void launch_ilu_solve(const RasDev& d, const double* r, double* z, int32_t* err, cudaStream_t s) {
  launch_ilu_solve_t<double>(d, r, z, err, s);
}

void launch_ilu_solve32(const RasDev& d, const float* r, float* z, int32_t* err, cudaStream_t s) {
  launch_ilu_solve_t<float>(d, r, z, err, s);
}

// shared-memory limits of every solve variant, set at context creation rather than in a
// captured launch
template <class T>
void solve_attrs_all() {
  RasDev d{};
  for (int P : {1, SOLVE_WIDE_MAX + 1})
    for (int w : {3, 7})
      for (int ring : {SOLVE_RING_HALF, SOLVE_RING_1, SOLVE_RING_2, SOLVE_RING_3, SOLVE_RING_4, SOLVE_RING_4F, SOLVE_RING_FULL}) {
        d.P = P;
        d.solve_warps = w;
        d.solve_ring = ring;
        solve_variant<T>(d, []<int NCW, int RB, bool WIDE>() {
          cudaFuncSetAttribute(k_ilu_solve<T, T, NCW, RB, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)solve_smem<T>(RB));
        });
      }
}

void launch_coarse_assemble(const CoarseDev& c, const double* val, const float* val32, cudaStream_t s) {
  const int64_t W = 2 * (int64_t)c.band + 1;
  cudaMemsetAsync(c.cband, 0, sizeof(double) * 25 * W * c.P, s);
  const int g = (int)((32 * (int64_t)c.nchunk + 255) / 256);
  if (val) k_coarse_chunks<double><<<g, 256, 0, s>>>(c.nchunk, c.cchunk_ptr, c.cseg_blk, val, c.cpart);
  else k_coarse_chunks<float><<<g, 256, 0, s>>>(c.nchunk, c.cchunk_ptr, c.cseg_blk, val32, c.cpart);
  k_coarse_dst<<<(int)((25 * (int64_t)c.ndst + 255) / 256), 256, 0, s>>>(c.ndst, c.cdst_ptr, c.cdst_idx, c.cpart,
                                                                          c.cband);
  count_launch();
  count_launch();
}

void launch_coarse_factor(const CoarseDev& c, int32_t* err, cudaStream_t s) {
  for (int kb = 0; kb < c.P; ++kb) {
    k_band_step<<<std::max(1, std::min(c.band, c.P - 1 - kb)), 256, 0, s>>>(c.P, c.band, kb, c.cband, c.cdinv, err);
    count_launch();
  }
  if (c.ainvT) {  // explicit inverse through the banded factors
    if (25 * (size_t)c.P * sizeof(double) <= 227 * 1024) {  // a block column of five unit vectors per CTA
      k_band_inv<<<c.P, 256, 25 * sizeof(double) * c.P, s>>>(c.P, c.band, c.cband, c.cdinv, c.ainvT);
    } else {  // one unit vector per CTA
      k_band_solve<<<5 * c.P, 256, sizeof(double) * 5 * c.P, s>>>(c.P, c.band, c.cband, c.cdinv, c.ainvT, 1);
    }
    count_launch();
  }
}

// y = A_c^{-1} Z^T r (left in crhs + 5P with the explicit inverse, in crhs otherwise)
void launch_coarse_solve(const CoarseDev& c, const double* r, cudaStream_t s) {
  k_coarse_restrict<<<c.P, 256, 0, s>>>(c.own_ptr, c.cpos, r, c.crhs);
  count_launch();
  const int nc = 5 * c.P;
  if (c.ainvT) {
    const int nchunk = (nc + GEMV_CHUNK - 1) / GEMV_CHUNK;
    k_coarse_gemv_part<<<dim3((nc + 127) / 128, nchunk), 128, 0, s>>>(nc, c.ainvT, c.crhs, c.cpart);
    k_coarse_gemv_sum<<<(nc + 127) / 128, 128, 0, s>>>(nc, nchunk, c.cpart, c.crhs + nc);
    count_launch();
    count_launch();
  } else {
    k_band_solve<<<1, 512, sizeof(double) * nc, s>>>(c.P, c.band, c.cband, c.cdinv, c.crhs, 0);
    count_launch();
  }
}

// z += Z y for the y of the last launch_coarse_solve
template <class TZ>
void launch_coarse_prolong(const CoarseDev& c, int64_t n, TZ* z, cudaStream_t s) {
  const int nc = 5 * c.P;
  int64_t g = (5 * n + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  k_coarse_prolong_add<TZ><<<(int)g, 256, 0, s>>>(n, c.owner, c.cpos, c.ainvT ? c.crhs + nc : c.crhs, z);
  count_launch();
}
template void launch_coarse_prolong<double>(const CoarseDev&, int64_t, double*, cudaStream_t);

void launch_coarse_y32(const CoarseDev& c, cudaStream_t s) {
  const int nc = 5 * c.P;
  k_coarse_to_f32<<<(nc + 255) / 256, 256, 0, s>>>(nc, c.ainvT ? c.crhs + nc : c.crhs, c.y32);
  count_launch();
}

void launch_coarse_prolong32(const CoarseDev& c, int64_t n, float* z, cudaStream_t s) {
  int64_t g = (5 * n + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  k_coarse_prolong_add32<<<(int)g, 256, 0, s>>>(n, c.owner, c.cpos, c.y32, z);
  count_launch();
}

template <class TZ>
void launch_coarse_apply_add(const CoarseDev& c, int64_t n, const double* r, TZ* z, cudaStream_t s) {
  launch_coarse_solve(c, r, s);
  launch_coarse_prolong<TZ>(c, n, z, s);
}
template void launch_coarse_apply_add<double>(const CoarseDev&, int64_t, const double*, double*, cudaStream_t);

// A Z segments: azval[s] = sum of the J blocks of segment s (one thread per entry)
template <class TV, class TA>
__global__ void k_az_build(int64_t nseg, const int32_t* __restrict__ az_blk, const TV* __restrict__ val,
                           TA* __restrict__ azval) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= 25 * nseg) return;
  const int64_t s = g / 25;
  const int e = (int)(g - 25 * s);
  double acc = 0.0;
  for (int32_t b = az_blk[s]; b < az_blk[s + 1]; ++b) acc += (double)val[25 * (int64_t)b + e];
  azval[g] = (TA)acc;
}

// t -= (A Z) y for the coarse solution y (cpos order): one thread per scalar row
template <class TA>
__global__ void k_az_sub(int64_t n, const int64_t* __restrict__ az_ptr, const int32_t* __restrict__ az_unit,
                         const int32_t* __restrict__ cpos, const TA* __restrict__ azval,
                         const double* __restrict__ y, double* __restrict__ t) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= 5 * n) return;
  const int64_t i = g / 5;
  const int rr = (int)(g - 5 * i);
  double acc = 0.0;
  for (int64_t s = az_ptr[i]; s < az_ptr[i + 1]; ++s) {
    const TA* A = azval + 25 * s + 5 * rr;
    const double* ys = y + 5 * (int64_t)cpos[az_unit[s]];
#pragma unroll
    for (int mm = 0; mm < 5; ++mm) acc = fma((double)A[mm], ys[mm], acc);
  }
  t[g] -= acc;
}

// the same with FP32 products for the mixed path, whose subdomain solve takes the result in
// FP32: out = (float)(t - (A Z) y), rows padded to eight values
__global__ void k_az_sub32(int64_t n, const int64_t* __restrict__ az_ptr, const int32_t* __restrict__ az_unit,
                           const int32_t* __restrict__ cpos, const float* __restrict__ azval,
                           const float* __restrict__ y, const double* __restrict__ t, float* __restrict__ out) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= 5 * n) return;
  const int64_t i = g / 5;
  const int rr = (int)(g - 5 * i);
  float acc = 0.0f;
  for (int64_t s = az_ptr[i]; s < az_ptr[i + 1]; ++s) {
    const float* A = azval + 25 * s + 5 * rr;
    const float* ys = y + 5 * (int64_t)cpos[az_unit[s]];
#pragma unroll
    for (int mm = 0; mm < 5; ++mm) acc = fmaf(A[mm], ys[mm], acc);
  }
  out[8 * i + rr] = (float)(t[g] - (double)acc);
}

// r in FP32 for the mixed path's subdomain solve, rows padded to eight values
__global__ void k_pack32(int64_t n, const double* __restrict__ r, float* __restrict__ out) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < 5 * n; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = g / 5;
    out[8 * i + (g - 5 * i)] = (float)r[g];
  }
}

void launch_pack32(int64_t n, const double* r, float* out, cudaStream_t s) {
  k_pack32<<<(unsigned)std::min<int64_t>((5 * n + 255) / 256, 152 * 8), 256, 0, s>>>(n, r, out);
  count_launch();
}

void launch_az_build(int64_t nseg, const int32_t* az_blk, const double* val, const float* val32, double* azval,
                     float* azval32, bool fp32, cudaStream_t s) {
  const unsigned g = (unsigned)((25 * nseg + 255) / 256);
  if (fp32) k_az_build<float, float><<<g, 256, 0, s>>>(nseg, az_blk, val32, azval32);
  else k_az_build<double, double><<<g, 256, 0, s>>>(nseg, az_blk, val, azval);
  count_launch();
}

void launch_az_sub(const CoarseDev& c, int64_t n, const int64_t* az_ptr, const int32_t* az_unit,
                   const double* azval, double* t, cudaStream_t s) {
  const double* y = c.ainvT ? c.crhs + 5 * (int64_t)c.P : c.crhs;
  k_az_sub<double><<<(unsigned)((5 * n + 255) / 256), 256, 0, s>>>(n, az_ptr, az_unit, c.cpos, azval, y, t);
  count_launch();
}

void launch_az_sub32(const CoarseDev& c, int64_t n, const int64_t* az_ptr, const int32_t* az_unit,
                     const float* azval, const double* t, float* out, cudaStream_t s) {
  k_az_sub32<<<(unsigned)((5 * n + 255) / 256), 256, 0, s>>>(n, az_ptr, az_unit, c.cpos, azval, c.y32, t, out);
  count_launch();
}

void coarse_init() {
  cudaFuncSetAttribute(k_band_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  cudaFuncSetAttribute(k_band_inv, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  const int row = FACTOR_CAP * 25;
  cudaFuncSetAttribute(k_ilu_factor<double, double, 512, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * row * 8);
  cudaFuncSetAttribute(k_ilu_factor<float, float, 512, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * row * 4);
  cudaFuncSetAttribute(k_ilu_factor<double, double, 256, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * row * 8);
  cudaFuncSetAttribute(k_ilu_factor<double, double, 256, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * row * 8);
  solve_attrs_all<double>();
  solve_attrs_all<float>();
}

}  // namespace seird
