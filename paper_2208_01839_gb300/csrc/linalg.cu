// BSR SpMV and the vector kernels of restarted right-preconditioned (F)GMRES
// with CGS2 orthogonalisation (Section 3.2: GMRES with right preconditioning;
// FGMRES when the preconditioner varies).  FP64 accumulation throughout;
// reductions are two-stage (per-CTA partials, then one CTA in fixed order), so
// every result is bitwise reproducible run to run.
#include <algorithm>
#include <cmath>

#include "kernels.cuh"

namespace seird {

namespace {

constexpr int NVMAX = 65;  // restart <= 64 -> at most 65 basis vectors

// (double)f on the integer pipe: GB300 converts at its FP64 rate, so a conversion costs as much
// as the FMA it feeds.  The exponent is rebiased (127 -> 1023) and the 23 fraction bits become
// the leading ones of 52; subnormals, infinities and NaNs take the conversion instruction.
__device__ __forceinline__ double widen(float f) {
  const uint32_t b = __float_as_uint(f), m = b & 0x7fffffffu;
  if (m - 0x00800000u >= 0x7f000000u && m != 0) return (double)f;
  const uint32_t hi = m ? (m >> 3) + 0x38000000u : 0u;
  return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(b << 29));
}

template <bool WIDEN>
__device__ __forceinline__ double ld_val(const double* p) {
  return __ldg(p);
}
template <bool WIDEN>
__device__ __forceinline__ double ld_val(const float* p) {
  return WIDEN ? widen(__ldg(p)) : (double)__ldg(p);
}

// y = A x (b == NULL) or y = b - A x, 5x5 blocks.  One thread per scalar output row (block
// row i, row r): all 32 lanes of every warp do useful FP64 work, 25 FMA per block per 5 threads.
// UNEVEN (a caller's own matrix): a warp takes as long as its longest row, so where a CTA's
// rows differ in length it takes them longest first, each row's rank counted on the integer
// pipe (rows of four to nine blocks, 1.95M blocks: 139.5 -> 102.8 us).  A mesh's rows are nearly
// all alike; for the Jacobian the sort only costs (2.0M nodes: 595 -> 601 us).
// WIDEN (FP32 values of a caller's matrix): widened by shifts instead of converted.  300,007
// rows of four to nine blocks 212 -> 202 us, 20,000 rows 27.5 -> 23.4; a mesh's Jacobian is
// slower that way (250k nodes 167.8 -> 170.6) and converts.
template <class VT, bool UNEVEN, bool WIDEN>
__global__ void __launch_bounds__(512) k_bsr_spmv(int64_t nrow, const int32_t* __restrict__ rp,
                                                  const int32_t* __restrict__ col, const VT* __restrict__ val,
                                                  const double* __restrict__ x, const double* __restrict__ b,
                                                  double* __restrict__ y) {
  int64_t i, g;  // block row and scalar row
  int r;
  if constexpr (UNEVEN) {
    __shared__ int32_t len[104];  // blockDim.x / 5 rows, at most 102
    __shared__ uint8_t order[104];
    const int R = blockDim.x / 5, q = threadIdx.x / 5;
    const int64_t i0 = blockIdx.x * (int64_t)R;
    const int nr = (int)(nrow - i0 < R ? nrow - i0 : R);
    r = threadIdx.x - 5 * q;
    if (threadIdx.x < nr) len[threadIdx.x] = __ldg(rp + i0 + threadIdx.x + 1) - __ldg(rp + i0 + threadIdx.x);
    __syncthreads();
    int mine = q;
    if (__syncthreads_or(threadIdx.x < nr && len[threadIdx.x] != len[0])) {
      if (threadIdx.x < nr) {
        const int l = len[threadIdx.x];
        int rank = 0;
        for (int k = 0; k < nr; ++k) rank += len[k] > l || (len[k] == l && k < (int)threadIdx.x);
        order[rank] = (uint8_t)threadIdx.x;
      }
      __syncthreads();
      if (q < nr) mine = order[q];
    }
    if (q >= nr) return;
    i = i0 + mine;
    g = 5 * i + r;
  } else {
    g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= 5 * nrow) return;
    i = g / 5;
    r = (int)(g - 5 * i);
  }
  const int32_t k0 = __ldg(rp + i), k1 = __ldg(rp + i + 1);
  double acc = 0.0;
  for (int32_t k = k0; k < k1; ++k) {
    const int64_t j = __ldg(col + k);
    const VT* v = val + 25 * (int64_t)k + 5 * r;
    const double* xj = x + 5 * j;
    acc = fma(ld_val<WIDEN>(v + 0), __ldg(xj + 0), acc);
    acc = fma(ld_val<WIDEN>(v + 1), __ldg(xj + 1), acc);
    acc = fma(ld_val<WIDEN>(v + 2), __ldg(xj + 2), acc);
    acc = fma(ld_val<WIDEN>(v + 3), __ldg(xj + 3), acc);
    acc = fma(ld_val<WIDEN>(v + 4), __ldg(xj + 4), acc);
  }
  y[g] = b ? b[g] - acc : acc;
}

// Mixed-precision SpMV: FP32 values and FP32 input, FP32 arithmetic, FP64 output (y = A x,
// or y = b - A x when b != NULL).
__global__ void __launch_bounds__(512) k_bsr_spmv32(int64_t nrow, const int32_t* __restrict__ rp,
                                                    const int32_t* __restrict__ col, const float* __restrict__ val,
                                                    const float* __restrict__ x, const double* __restrict__ b,
                                                    double* __restrict__ y) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= 5 * nrow) return;
  const int64_t i = g / 5;
  const int r = (int)(g - 5 * i);
  const int32_t k0 = __ldg(rp + i), k1 = __ldg(rp + i + 1);
  float acc = 0.f;
  for (int32_t k = k0; k < k1; ++k) {
    const int64_t j = __ldg(col + k);
    const float* v = val + 25 * (int64_t)k + 5 * r;
    const float* xj = x + 5 * j;
#pragma unroll
    for (int c = 0; c < 5; ++c) acc = fmaf(__ldg(v + c), __ldg(xj + c), acc);
  }
  y[g] = b ? b[g] - (double)acc : (double)acc;
}

// x += sum_k coef[k] Z_k with FP32 Z: the sum is formed in FP32, added in FP64
__global__ void k_multi_axpy32(int64_t len, int nv, const float* __restrict__ Z, int64_t ld,
                               const double* __restrict__ coef, double* __restrict__ x) {
  __shared__ float cs[NVMAX];
  for (int k = threadIdx.x; k < nv; k += blockDim.x) cs[k] = (float)coef[k];
  __syncthreads();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
    float v = 0.f;
    for (int k = 0; k < nv; ++k) v = fmaf(cs[k], Z[k * ld + i], v);
    x[i] += (double)v;
  }
}

// valT = J^T on the same (structurally symmetric) block pattern: block k = (i,j)
// of J^T is the transpose of block tpos[k] = (j,i) of J
__global__ void k_bsr_transpose(int64_t nnzb, const int32_t* __restrict__ tpos, const double* __restrict__ val,
                                double* __restrict__ valT) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < 25 * nnzb;
       g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = g / 25;
    const int e = (int)(g - 25 * k), rr = e / 5, cc = e % 5;
    valT[g] = val[25 * (int64_t)tpos[k] + 5 * cc + rr];
  }
}

// *flag |= 1 when a and b differ in any bit pattern (so NaNs and signed zeros count as they are stored)
__global__ void k_differs(int64_t len, const double* __restrict__ a, const double* __restrict__ b, int* flag) {
  bool d = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
    d |= __double_as_longlong(a[i]) != __double_as_longlong(b[i]);
  if (__any_sync(0xffffffffu, d) && (threadIdx.x & 31) == 0) atomicOr(flag, 1);
}

__global__ void k_add32(int64_t len, const float* __restrict__ u, float* __restrict__ z) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
    z[i] += u[i];
}

__global__ void k_f32_to_f64(int64_t n, const float* __restrict__ a, double* __restrict__ b) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    b[i] = (double)a[i];
}

template <int NT>
__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x < 32) {
    r = threadIdx.x < NT / 32 ? sh[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  __syncthreads();
  return r;  // valid in thread 0
}

// partial[cta] = sum over the CTA's slice of x^2
__global__ void __launch_bounds__(256) k_norm2_partial(int64_t len, const double* __restrict__ x,
                                                       double* __restrict__ partial) {
  __shared__ double sh[8];
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = x[i];
    s += v * v;
  }
  s = block_sum<256>(s, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// out[k] (+)= sum_cta partial[cta * stride + k], fixed order; CTA k sums column k (one CTA
// for all columns took 15.7 us for 456 partials of 16 columns, which is 2.5 us this way)
__global__ void __launch_bounds__(256) k_reduce_cols(int grid, int stride, const double* __restrict__ partial,
                                                     double* out, int add) {
  __shared__ double sh[8];
  const int k = blockIdx.x;
  double s = 0.0;
  for (int c = threadIdx.x; c < grid; c += blockDim.x) s += partial[(int64_t)c * stride + k];
  s = block_sum<256>(s, sh);
  if (threadIdx.x == 0) out[k] = add ? out[k] + s : s;
}

constexpr int KPW = (NVMAX + 7) / 8;  // dot products per warp

__device__ __forceinline__ void cp_async8(void* dst, const void* src, bool valid) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  const int n = valid ? 8 : 0;  // src-size 0: nothing is read, the destination is zero-filled
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// CGS passes with double-buffered tiles: while tile t is consumed from shared
// memory, the basis entries (and w) of tile t+1 stream in through cp.async, so
// the FP64 pipe does not wait for the loads.  T entries per tile (256, or 128
// when many basis vectors would not fit twice).
// mode 0: partial[cta][k] = sum V_k . w ; mode 1: w -= V h, then the dots with w_new
template <int MODE, int T>
__global__ void __launch_bounds__(256) k_cgs_db(int64_t len, int nv, const double* __restrict__ V, int64_t ld,
                                                const double* __restrict__ h, double* __restrict__ w,
                                                double* __restrict__ partial) {
  extern __shared__ double smem[];
  double* hs = smem;                 // [NVMAX + 7]
  double* wt = hs + NVMAX + 7;       // [T] current w tile (after the update)
  double* bufs = wt + T;             // [2][nv + 1][T]: basis tiles and the incoming w tile
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int nvb = nv + 1;
  if (MODE == 1)
    for (int k = tid; k < nv; k += blockDim.x) hs[k] = h[k];
  double acc[KPW];
#pragma unroll
  for (int q = 0; q < KPW; ++q) acc[q] = 0.0;
  const int64_t ntile = (len + T - 1) / T;
  auto load = [&](int64_t tile, int b) {
    double* dst = bufs + (size_t)b * nvb * T;
    const int64_t base = tile * T;
    for (int idx = tid; idx < nvb * T; idx += blockDim.x) {
      const int k = idx / T, e = idx - k * T;
      const int64_t i = base + e;
      const bool ok = i < len;
      const double* src = (k < nv ? V + k * ld : w) + (ok ? i : 0);
      cp_async8(dst + idx, src, ok);
    }
  };
  int64_t tile = blockIdx.x;
  if (tile < ntile) load(tile, 0);
  cp_async_commit();
  for (int b = 0; tile < ntile; tile += gridDim.x, b ^= 1) {
    if (tile + gridDim.x < ntile) load(tile + gridDim.x, b ^ 1);
    cp_async_commit();
    cp_async_wait1();  // the current tile's group has landed (this thread's copies)
    __syncthreads();   // ... and everyone else's
    const double* Vt = bufs + (size_t)b * nvb * T;
    const double* wsrc = Vt + (size_t)nv * T;
    for (int e = tid; e < T; e += blockDim.x) {
      double wi = wsrc[e];
      if (MODE == 1) {
        for (int k = 0; k < nv; ++k) wi = fma(-hs[k], Vt[k * T + e], wi);
        const int64_t i = tile * T + e;
        if (i < len) w[i] = wi;
      }
      wt[e] = wi;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < KPW; ++q) {
      const int k = wp + 8 * q;
      if (k < nv) {
        double s = acc[q];
#pragma unroll
        for (int e = lane; e < T; e += 32) s = fma(Vt[k * T + e], wt[e], s);
        acc[q] = s;
      }
    }
    __syncthreads();  // buffer b is refilled two tiles later
  }
#pragma unroll
  for (int q = 0; q < KPW; ++q) {
    const int k = wp + 8 * q;
    double s = acc[q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0 && k < nv) partial[blockIdx.x * (int64_t)NVMAX + k] = s;
  }
}

inline size_t cgs_db_smem(int nv, int T) { return sizeof(double) * (NVMAX + 7 + T + 2 * (size_t)(nv + 1) * T); }

// tile entries per CTA step: the caller's choice (128 or 256; 0 = by length and depth), 128
// whenever 256 would not fit twice in shared memory, and 64 for vectors that would otherwise
// leave SMs without a tile (5445 entries, 16 vectors: 13.5 us a pass with 22 CTAs of 256)
inline int cgs_tile(int64_t len, int nv, int want = 0) {
  if (want == 0 && len <= 152 * 128) return 64;
  if (nv > 27) return 128;
  return want == 128 ? 128 : 256;
}
// CTAs of a pass: no more than there are tiles (the rest would only add zeros to the sums)
inline int cgs_grid(int64_t len, int T, int grid) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(grid, (len + T - 1) / T));
}
template <int MODE>
void launch_cgs_db(int T, int64_t len, int nv, const double* V, int64_t ld, const double* h, double* w,
                   double* partial, int grid, cudaStream_t s) {
  const size_t sm = cgs_db_smem(nv, T);
  if (T == 256) k_cgs_db<MODE, 256><<<grid, 256, sm, s>>>(len, nv, V, ld, h, w, partial);
  else if (T == 128) k_cgs_db<MODE, 128><<<grid, 256, sm, s>>>(len, nv, V, ld, h, w, partial);
  else k_cgs_db<MODE, 64><<<grid, 256, sm, s>>>(len, nv, V, ld, h, w, partial);
}

// second CGS pass update and ||w||^2 without staging: every thread needs only its
// own entries of the basis vectors, so they go straight to registers
__global__ void __launch_bounds__(256) k_cgs_update_norm(int64_t len, int nv, const double* __restrict__ V,
                                                         int64_t ld, const double* __restrict__ h,
                                                         double* __restrict__ w, double* __restrict__ partial) {
  __shared__ double hs[NVMAX];
  __shared__ double sh[8];
  for (int k = threadIdx.x; k < nv; k += blockDim.x) hs[k] = h[k];
  __syncthreads();
  double nrm = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
    double a0 = w[i], a1 = 0.0;
    int k = 0;
    for (; k + 1 < nv; k += 2) {
      a0 = fma(-hs[k], __ldg(V + k * ld + i), a0);
      a1 = fma(-hs[k + 1], __ldg(V + (k + 1) * ld + i), a1);
    }
    if (k < nv) a0 = fma(-hs[k], __ldg(V + k * ld + i), a0);
    const double wi = a0 + a1;
    w[i] = wi;
    nrm = fma(wi, wi, nrm);
  }
  nrm = block_sum<256>(nrm, sh);
  if (threadIdx.x == 0) partial[blockIdx.x * (int64_t)NVMAX] = nrm;
}

// y = x * a (invert: a := 1/a), a read from device memory; a == 0 gives y = 0
__global__ void k_scale(int64_t len, const double* __restrict__ x, const double* __restrict__ ap, int invert,
                        double* __restrict__ y) {
  double a = *ap;
  if (invert) a = a != 0.0 ? 1.0 / a : 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = a * x[i];
}

__global__ void k_axpby(int64_t len, double a, const double* __restrict__ x, double b, const double* __restrict__ y,
                        double* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = a * x[i] + b * y[i];
}

// x += sum_k coef[k] Z_k
__global__ void k_multi_axpy(int64_t len, int nv, const double* __restrict__ Z, int64_t ld,
                             const double* __restrict__ coef, double* __restrict__ x) {
  __shared__ double cs[NVMAX];
  for (int k = threadIdx.x; k < nv; k += blockDim.x) cs[k] = coef[k];
  __syncthreads();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
    double v = x[i];
    for (int k = 0; k < nv; ++k) v = fma(cs[k], Z[k * ld + i], v);
    x[i] = v;
  }
}

// GMRES small state layout in gm (ldh = restart+1):
//   H[ldh*restart] column-major (H[row + ldh*col]), cs[restart], sn[restart], g[ldh], y[restart]
// Column j of H gets hcol[0..j] and hnext; previous rotations are applied, a new
// rotation annihilates H[j+1, j]; |g[j+1]| (the residual norm) goes to *out_res.
// In a captured restart cycle (cc.ctl != NULL) the kernel also takes the convergence
// decision of the iteration: cc.ctl[0] = iterations run, cc.ctl[2] = outcome (0 go on,
// 1 converged or breakdown, 2 past dtol or not finite), cc.ctl[1] = iteration limit of
// the cycle; cc.tol = {tolerance, dtol * ||b||}.  It arms the conditional node of the
// next iteration (cc.next) only while the outcome is 0 and the limit is not reached.
__global__ void k_givens(int j, double* gm, const double* __restrict__ h1, const double* __restrict__ h2,
                         const double* __restrict__ hnext_sq, int ldh, double* out_res, CycleCtl cc) {
  // the warp brings the column, the rotations and the scalars on chip at once; the chain of
  // rotations is one thread's, and the warp writes the column (one thread alone took 9 us at
  // j = 16, nearly all of it waiting for its loads one after the other)
  __shared__ double col[NVMAX + 1], rc[NVMAX], rs[NVMAX];
  const int restart = ldh - 1, lane = threadIdx.x;
  double* H = gm;
  double* cs = H + (int64_t)ldh * restart;
  double* sn = cs + restart;
  double* g = sn + restart;
  for (int k = lane; k <= j; k += 32) {
    col[k] = h1[k] + h2[k];  // CGS2: both passes' coefficients
    if (k < j) {
      rc[k] = cs[k];
      rs[k] = sn[k];
    }
  }
  const double hn = sqrt(fmax(*hnext_sq, 0.0));
  const double gj = g[j];
  __syncwarp();
  if (lane == 0) {
    double a = col[0];
    for (int k = 0; k < j; ++k) {
      const double b = col[k + 1];
      col[k] = rc[k] * a + rs[k] * b;
      a = -rs[k] * a + rc[k] * b;
    }
    const double b = hn;
    const double rr = hypot(a, b);
    double c = 1.0, s = 0.0;
    if (rr != 0.0) {
      c = a / rr;
      s = b / rr;
    }
    cs[j] = c;
    sn[j] = s;
    col[j] = rr;
    col[j + 1] = 0.0;
    g[j] = c * gj;
    const double gn = -s * gj;
    g[j + 1] = gn;
    const double res = fabs(gn);
    out_res[0] = res;
    out_res[1] = hn;
    if (cc.ctl) {
      int outcome = 0;
      if (!(res <= cc.tol[1]) || !isfinite(res)) outcome = 2;
      else if (res <= cc.tol[0] || hn == 0.0) outcome = 1;
      cc.ctl[0] = j + 1;
      cc.ctl[2] = outcome;
      if (cc.has_next) cudaGraphSetConditional(cc.next, (outcome == 0 && j + 1 < cc.ctl[1]) ? 1u : 0u);
    }
  }
  __syncwarp();
  for (int k = lane; k <= j + 1; k += 32) H[k + (int64_t)ldh * j] = col[k];
}

// y = H(0:k,0:k)^{-1} g(0:k) by back substitution: the CTA brings the triangle on chip, one
// thread solves
__global__ void __launch_bounds__(256) k_hsolve(int k, double* gm, int ldh) {
  extern __shared__ double hs[];  // [k][k] column-major, then g
  const int restart = ldh - 1;
  const double* H = gm;
  double* g = gm + (int64_t)ldh * restart + 2 * restart;
  double* y = g + ldh;
  for (int q = threadIdx.x; q < k * k; q += blockDim.x) hs[q] = H[q % k + (int64_t)ldh * (q / k)];
  double* v = hs + k * k;
  for (int q = threadIdx.x; q < k; q += blockDim.x) v[q] = g[q];
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int i = k - 1; i >= 0; --i) {
    double t = v[i];
    for (int c = i + 1; c < k; ++c) t -= hs[i + k * c] * v[c];
    const double d = hs[i + k * i];
    t = d != 0.0 ? t / d : 0.0;
    v[i] = t;
    y[i] = t;
  }
}

__global__ void k_gather5(int64_t n, const int32_t* __restrict__ idx, const double* __restrict__ src,
                          double* __restrict__ dst, const double* __restrict__ src2, double* __restrict__ dst2) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < 5 * n; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = g / 5;
    const int64_t f = 5 * (int64_t)idx[k] + (g - 5 * k);
    dst[g] = src[f];
    if (src2) dst2[g] = src2[f];
  }
}

__global__ void k_scatter5(int64_t n, const int32_t* __restrict__ idx, const double* __restrict__ src,
                           double* __restrict__ dst) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < 5 * n; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = g / 5;
    dst[5 * (int64_t)idx[k] + (g - 5 * k)] = src[g];
  }
}

inline int grid_for(int64_t len, int tb = 256, int cap = 152 * 8) {
  int64_t g = (len + tb - 1) / tb;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

template <class VT>
void launch_spmv(int64_t nrow, const int32_t* rp, const int32_t* col, const VT* val, const double* x, double* y,
                 cudaStream_t s, int tb, const double* b) {
  if (nrow <= 0) return;
  k_bsr_spmv<VT, false, false><<<(unsigned)((5 * nrow + tb - 1) / tb), tb, 0, s>>>(nrow, rp, col, val, x, b, y);
  count_launch();
}
template <class VT>
void launch_spmv_uneven(int64_t nrow, const int32_t* rp, const int32_t* col, const VT* val, const double* x, double* y,
                        cudaStream_t s) {
  if (nrow <= 0) return;
  const int tb = 256, R = tb / 5;
  // up to one wave of CTAs the launch lasts as long as its longest row whatever their order
  // (a few thousand rows: 13.5 us plain, 14.3 sorted)
  constexpr bool W = sizeof(VT) == 4;
  if (nrow <= 152 * 8 * (int64_t)R)
    k_bsr_spmv<VT, false, W><<<(unsigned)((5 * nrow + tb - 1) / tb), tb, 0, s>>>(nrow, rp, col, val, x, nullptr, y);
  else
    k_bsr_spmv<VT, true, W><<<(unsigned)((nrow + R - 1) / R), tb, 0, s>>>(nrow, rp, col, val, x, nullptr, y);
  count_launch();
}
template void launch_spmv<double>(int64_t, const int32_t*, const int32_t*, const double*, const double*, double*,
                                  cudaStream_t, int, const double*);
template void launch_spmv<float>(int64_t, const int32_t*, const int32_t*, const float*, const double*, double*,
                                 cudaStream_t, int, const double*);
template void launch_spmv_uneven<double>(int64_t, const int32_t*, const int32_t*, const double*, const double*, double*,
                                         cudaStream_t);
template void launch_spmv_uneven<float>(int64_t, const int32_t*, const int32_t*, const float*, const double*, double*,
                                        cudaStream_t);

void launch_spmv32(int64_t nrow, const int32_t* rp, const int32_t* col, const float* val, const float* x, double* y,
                   cudaStream_t s, int tb, const double* b) {
  if (nrow <= 0) return;
  k_bsr_spmv32<<<(5 * nrow + tb - 1) / tb, tb, 0, s>>>(nrow, rp, col, val, x, b, y);
  count_launch();
}

void launch_multi_axpy32(int64_t len, int nv, const float* Zs, int64_t ld, const double* coef, double* x,
                         cudaStream_t s) {
  k_multi_axpy32<<<grid_for(len), 256, 0, s>>>(len, nv, Zs, ld, coef, x);
  count_launch();
}

void launch_bsr_transpose(int64_t nnzb, const int32_t* tpos, const double* val, double* valT, cudaStream_t s) {
  k_bsr_transpose<<<grid_for(25 * nnzb), 256, 0, s>>>(nnzb, tpos, val, valT);
  count_launch();
}

void launch_differs(int64_t len, const double* a, const double* b, int* flag, cudaStream_t s) {
  cudaMemsetAsync(flag, 0, sizeof(int), s);
  k_differs<<<grid_for(len), 256, 0, s>>>(len, a, b, flag);
  count_launch();
}

void launch_add32(int64_t len, const float* u, float* z, cudaStream_t s) {
  k_add32<<<grid_for(len), 256, 0, s>>>(len, u, z);
  count_launch();
}

void launch_f32_to_f64(int64_t n, const float* src, double* dst, cudaStream_t s) {
  k_f32_to_f64<<<grid_for(n), 256, 0, s>>>(n, src, dst);
  count_launch();
}

void launch_norm2(int64_t len, const double* x, double* partial, int grid, double* out, cudaStream_t s) {
  const int g = cgs_grid(len, 256, grid);
  k_norm2_partial<<<g, 256, 0, s>>>(len, x, partial);
  k_reduce_cols<<<1, 256, 0, s>>>(g, 1, partial, out, 0);
  count_launch();
  count_launch();
}

void launch_mdot(int64_t len, int nv, const double* V, int64_t ld, const double* w, double* partial, int grid,
                 double* out, cudaStream_t s, int tile) {
  const int T = cgs_tile(len, nv, tile), g = cgs_grid(len, T, grid);
  launch_cgs_db<0>(T, len, nv, V, ld, nullptr, const_cast<double*>(w), partial, g, s);
  k_reduce_cols<<<nv, 256, 0, s>>>(g, NVMAX, partial, out, 0);
  count_launch();
  count_launch();
}

// first CGS pass update fused with the second pass's dot products (to out)
void launch_update_mdot(int64_t len, int nv, const double* V, int64_t ld, const double* h, double* w,
                        double* partial, int grid, double* out, cudaStream_t s, int tile) {
  const int T = cgs_tile(len, nv, tile), g = cgs_grid(len, T, grid);
  launch_cgs_db<1>(T, len, nv, V, ld, h, w, partial, g, s);
  k_reduce_cols<<<nv, 256, 0, s>>>(g, NVMAX, partial, out, 0);
  count_launch();
  count_launch();
}

void launch_update_norm(int64_t len, int nv, const double* V, int64_t ld, const double* h, double* w,
                        double* partial, int grid, double* out, cudaStream_t s) {
  const int g = cgs_grid(len, 256, grid);
  k_cgs_update_norm<<<g, 256, 0, s>>>(len, nv, V, ld, h, w, partial);
  k_reduce_cols<<<1, 256, 0, s>>>(g, NVMAX, partial, out, 0);
  count_launch();
  count_launch();
}

void cgs_init() {
  const int mx = 227 * 1024;
  cudaFuncSetAttribute(k_cgs_db<0, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
  cudaFuncSetAttribute(k_cgs_db<1, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
  cudaFuncSetAttribute(k_cgs_db<0, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
  cudaFuncSetAttribute(k_cgs_db<1, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
  cudaFuncSetAttribute(k_cgs_db<0, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
  cudaFuncSetAttribute(k_cgs_db<1, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
}

void launch_reduce_cols(int grid, int nv, const double* partial, double* out, int add, cudaStream_t s) {
  k_reduce_cols<<<nv, 256, 0, s>>>(grid, NVMAX, partial, out, add);
  count_launch();
}

void launch_scale(int64_t len, const double* x, const double* alpha_ptr, int invert, double* y, cudaStream_t s) {
  k_scale<<<grid_for(len), 256, 0, s>>>(len, x, alpha_ptr, invert, y);
  count_launch();
}

void launch_axpby(int64_t len, double a, const double* x, double b, const double* y, double* out, cudaStream_t s) {
  k_axpby<<<grid_for(len), 256, 0, s>>>(len, a, x, b, y, out);
  count_launch();
}

void launch_multi_axpy(int64_t len, int nv, const double* Zs, int64_t ld, const double* coef, double* x,
                       cudaStream_t s) {
  k_multi_axpy<<<grid_for(len), 256, 0, s>>>(len, nv, Zs, ld, coef, x);
  count_launch();
}

void launch_givens(int j, double* gm, const double* h1, const double* h2, const double* hnext, int ldh,
                   double* out_res, cudaStream_t s, const CycleCtl& cc) {
  k_givens<<<1, 32, 0, s>>>(j, gm, h1, h2, hnext, ldh, out_res, cc);
  count_launch();
}

void launch_hsolve(int k, double* gm, int ldh, cudaStream_t s) {
  k_hsolve<<<1, 256, sizeof(double) * (size_t)k * (k + 1), s>>>(k, gm, ldh);
  count_launch();
}

void launch_gather5(int64_t n, const int32_t* idx, const double* src, double* dst, cudaStream_t s,
                    const double* src2, double* dst2) {
  k_gather5<<<grid_for(5 * n), 256, 0, s>>>(n, idx, src, dst, src2, dst2);
  count_launch();
}

void launch_scatter5(int64_t n, const int32_t* idx, const double* src, double* dst, cudaStream_t s) {
  k_scatter5<<<grid_for(5 * n), 256, 0, s>>>(n, idx, src, dst);
  count_launch();
}

}  // namespace seird
