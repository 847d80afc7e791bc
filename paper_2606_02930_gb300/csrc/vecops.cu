// Krylov vector kernels (Arnoldi step, block axpy, norms, scaling), the MPO
// mixing kernel, small trace/site-operator kernels and the device-side GMRES
// control (Givens QR of the Hessenberg matrix) of the local solves.
//
// All reductions are two-stage with a grid size fixed by the vector length,
// and the second stage sums the partials in block order, so results are
// bitwise reproducible run to run.
#include "common.cuh"

namespace ite {
namespace {

constexpr int VT = 256;          // threads per block of the vector kernels
constexpr int MAXV = 32;         // largest Krylov basis handled

int grid_for(long long n) {
  long long g = (n + VT - 1) / VT;
  if (g > 608) g = 608;          // 4 blocks per SM on 152 SMs
  if (g < 1) g = 1;
  return (int)g;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// block-wide sum of one double; result valid in thread 0
__device__ double block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (wid == 0) {
    r = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : 0.0;
    r = warp_sum(r);
  }
  __syncthreads();
  return r;
}

__global__ void k_copy(cplx* y, const cplx* x, long long n) {
  for (long long e = blockIdx.x * (long long)VT + threadIdx.x; e < n; e += (long long)gridDim.x * VT)
    y[e] = x[e];
}

__global__ void k_zero(cplx* y, long long n) {
  for (long long e = blockIdx.x * (long long)VT + threadIdx.x; e < n; e += (long long)gridDim.x * VT)
    y[e] = cmake(0.0, 0.0);
}

__global__ void k_axpby(cplx* y, const cplx* x, cplx a, cplx b, long long n) {
  for (long long e = blockIdx.x * (long long)VT + threadIdx.x; e < n; e += (long long)gridDim.x * VT)
    y[e] = cadd(cmul(a, x[e]), cmul(b, y[e]));
}

// out[i] = sum over the nblk partial rows of column i: warp i takes column
// i, its lanes sum rows lane, lane + 32, ... in order and a fixed shuffle tree
// adds the lanes, so the order of the sum is fixed and each lane issues its
// loads together (a single thread summing the rows one by one waited on each
// L2 load in turn, tens of microseconds per call).
__global__ void k_reduce_cplx(const cplx* partial, int nblk, int nv, cplx* out, const int* active) {
  if (active && *active == 0) return;
  const int i = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (i >= nv) return;
  double sr = 0.0, si = 0.0;
  for (int b = lane; b < nblk; b += 32) {
    const cplx v = partial[(long long)b * nv + i];
    sr += v.x;
    si += v.y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sr += __shfl_xor_sync(0xffffffffu, sr, o);
    si += __shfl_xor_sync(0xffffffffu, si, o);
  }
  if (lane == 0) out[i] = cmake(sr, si);
}

__global__ void k_block_axpy(const cplx* V, long long ldv, int nv, const int* nv_dev,
                             const cplx* h, double sign, cplx* w, long long n, const int* active) {
  if (active && *active == 0) return;
  __shared__ cplx hs[MAXV];
  int m = nv;
  if (nv_dev && *nv_dev < m) m = *nv_dev;
  if (threadIdx.x < m) hs[threadIdx.x] = cscale(h[threadIdx.x], sign);
  __syncthreads();
  for (long long e = blockIdx.x * (long long)VT + threadIdx.x; e < n; e += (long long)gridDim.x * VT) {
    cplx acc = w[e];
    for (int i = 0; i < m; ++i) cfma(acc, hs[i], V[(long long)i * ldv + e]);
    w[e] = acc;
  }
}

__global__ void k_norm2_partial(const cplx* x, long long n, double* partial, const int* active) {
  if (active && *active == 0) return;
  __shared__ double sh[32];
  double acc = 0.0;
  for (long long e = blockIdx.x * (long long)VT + threadIdx.x; e < n; e += (long long)gridDim.x * VT) {
    const cplx v = x[e];
    acc = fma(v.x, v.x, acc);
    acc = fma(v.y, v.y, acc);
  }
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// *out = sum of the nblk partials, by one warp in the fixed order of
// k_reduce_cplx
__global__ void k_reduce_real(const double* partial, int nblk, double* out, const int* active) {
  if (active && *active == 0) return;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x >= 32) return;
  double s = 0.0;
  for (int b = lane; b < nblk; b += 32) s += partial[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) *out = s;
}

__global__ void k_scale_dev(cplx* y, const double* scale, long long n, const int* active) {
  if (active && *active == 0) return;
  const double s = *scale;
  for (long long e = blockIdx.x * (long long)VT + threadIdx.x; e < n; e += (long long)gridDim.x * VT)
    y[e] = cscale(y[e], s);
}

// L is D x m x n, R is D x n x m; sum_{w,b,c} L[w][b][c] R[w][c][b]
__global__ void k_env_trace(const cplx* L, const cplx* R, int D, int m, int n, cplx* partial) {
  __shared__ double sh[32];
  const long long tot = (long long)D * m * n;
  cplx acc = cmake(0.0, 0.0);
  for (long long e = blockIdx.x * (long long)VT + threadIdx.x; e < tot; e += (long long)gridDim.x * VT) {
    const long long w = e / ((long long)m * n);
    const long long rem = e - w * (long long)m * n;
    const long long b = rem / n, c = rem - b * n;
    cfma(acc, L[e], R[(w * n + c) * m + b]);
  }
  const double re = block_sum(acc.x, sh);
  const double im = block_sum(acc.y, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = cmake(re, im);
}

__global__ void k_site_op(const cplx* O, const cplx* K, cplx* Kout, int chl, int d, int chr) {
  const long long tot = (long long)chl * d * chr;
  for (long long e = blockIdx.x * (long long)VT + threadIdx.x; e < tot; e += (long long)gridDim.x * VT) {
    const long long a = e / ((long long)d * chr);
    const long long rem = e - a * d * chr;
    const int sp = (int)(rem / chr);
    const long long b = rem - (long long)sp * chr;
    cplx acc = cmake(0.0, 0.0);
    for (int s = 0; s < d; ++s) cfma(acc, O[sp * d + s], K[(a * d + s) * chr + b]);
    Kout[e] = acc;
  }
}

// ------------------------------------------------------------------ mixing
constexpr int MIX_MAX = 128;   // largest row/column count of a mixing matrix

constexpr int MIX_NNZ = 1024;  // entries staged in shared memory
constexpr int MIX_Q = 32;      // values of q per block
constexpr int MIX_G = 8;       // row groups per block

// One block per (p, 32 values of q): thread (q, g) forms the rows g, g + 8, ...
// The entries (value and input offset) are staged in shared memory, so that a
// term costs one load of the input and its products; real entries (every spin
// or fermion operator in use) take two FP64 products per term instead of four.
// (One thread for all rows of a (p, q), reading the entries from global memory
// one after the other, took 20-23 us at every size: 32 blocks and a chain of
// dependent loads at chi = 64, the FP64 pipe at chi = 256.)
__global__ void __launch_bounds__(MIX_Q* MIX_G)
k_mix(MixPlan pl, MixStrides s, int P, int Q, const cplx* in, long long iP, long long iQ, cplx* out,
      long long oP, long long oQ) {
  __shared__ long long ioff[MIX_MAX], ooff[MIX_MAX];
  __shared__ int rp[MIX_MAX + 1];
  __shared__ long long soff[MIX_NNZ];
  __shared__ cplx sval[MIX_NNZ];
  const int tid = threadIdx.x;
  for (int j = tid; j < pl.ncols; j += blockDim.x) {
    const int j2 = j % pl.cdim[2], j1 = (j / pl.cdim[2]) % pl.cdim[1], j0 = j / (pl.cdim[2] * pl.cdim[1]);
    ioff[j] = j0 * s.ic[0] + j1 * s.ic[1] + j2 * s.ic[2];
  }
  for (int k = tid; k < pl.nrows; k += blockDim.x) {
    const int k2 = k % pl.rdim[2], k1 = (k / pl.rdim[2]) % pl.rdim[1], k0 = k / (pl.rdim[2] * pl.rdim[1]);
    ooff[k] = k0 * s.oc[0] + k1 * s.oc[1] + k2 * s.oc[2];
  }
  for (int k = tid; k <= pl.nrows; k += blockDim.x) rp[k] = pl.row_ptr[k];
  __syncthreads();
  const bool staged = pl.nnz <= MIX_NNZ;
  int real = staged;
  if (staged)
    for (int e = tid; e < pl.nnz; e += blockDim.x) {
      const cplx v = pl.val[e];
      sval[e] = v;
      soff[e] = ioff[pl.col[e]];
      if (v.y != 0.0) real = 0;
    }
  real = __syncthreads_and(real);
  const int qt = (Q + MIX_Q - 1) / MIX_Q;
  const long long tiles = (long long)P * qt;
  const int ql = tid % MIX_Q, g = tid / MIX_Q;
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    const long long p = t / qt, q = (t - p * qt) * MIX_Q + ql;
    if (q >= Q) continue;
    const cplx* ib = in + p * iP + q * iQ;
    cplx* ob = out + p * oP + q * oQ;
    for (int k = g; k < pl.nrows; k += MIX_G) {
      cplx acc = cmake(0.0, 0.0);
      const int e1 = rp[k + 1];
      if (real) {
#pragma unroll 4
        for (int e = rp[k]; e < e1; ++e) {
          const double v = sval[e].x;
          const cplx x = ib[soff[e]];
          acc.x = fma(v, x.x, acc.x);
          acc.y = fma(v, x.y, acc.y);
        }
      } else if (staged) {
#pragma unroll 4
        for (int e = rp[k]; e < e1; ++e) cfma(acc, sval[e], ib[soff[e]]);
      } else {
        for (int e = rp[k]; e < e1; ++e) cfma(acc, pl.val[e], ib[ioff[__ldg(pl.col + e)]]);
      }
      ob[ooff[k]] = acc;
    }
  }
}

// ------------------------------------------------------------------ Arnoldi step
// One Arnoldi step of the local solve's GMRES (classical Gram-Schmidt twice) in
// three kernels and a scaling:
//   k_arnoldi_dot   h1 = V^H w
//   k_arnoldi_mid   w -= V h1, h2 = V^H w
//   k_arnoldi_end   w -= V h2, |w|^2, then the Givens update of the step
// Each sum ends in the block that finishes last (a counter in device memory),
// which adds the other blocks' shares in a fixed order, so no kernel is launched
// to add up 600 numbers; w is read and written by the same thread throughout.
// Bound: the launches and the FP64 adds of the reductions.  A warp-wide sum of
// one double takes five adds of 16 clocks on the SM's FP64 pipe, so eight sums
// are reduced together, halving what a lane holds at each exchange (9 adds
// instead of 40).  Eleven kernels per step before (n = 16384, chi = 64: 13 us a
// dot, 12 us for the Givens update by one thread reading global memory); now
// 9.6, 10.8 and 17 us for the three at chi = 64, the last 10 of them the chain of
// the Givens update.  GMRES(10): 1.91 -> 1.56 ms at chi = 64.
constexpr int AT = 128;          // threads per block
constexpr int AW = AT / 32;

int arnoldi_grid(long long n) {
  long long g = (n + AT - 1) / AT;
  return (int)(g > 608 ? 608 : g < 1 ? 1 : g);
}

// sh[warp][2 i], sh[warp][2 i + 1] = this warp's share of conj(V_i) . w over the
// elements of its threads
__device__ __forceinline__ void dot_shares(const cplx* V, long long ldv, int nv, const cplx* w,
                                           long long n, double (*sh)[2 * MAXV + 6]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int i0 = 0; i0 < nv; i0 += 4) {
    cplx acc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] = cmake(0.0, 0.0);
    for (long long e = blockIdx.x * (long long)AT + threadIdx.x; e < n; e += (long long)gridDim.x * AT) {
      const cplx we = w[e];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u < nv) cfma_conj(acc[u], V[(long long)(i0 + u) * ldv + e], we);
    }
    double v[8];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[2 * u] = acc[u].x;
      v[2 * u + 1] = acc[u].y;
    }
    const double r = warp_sum8(v);
    if ((lane & 3) == 0) sh[wid][2 * i0 + (lane >> 2)] = r;
  }
}

// w -= sum_i h_i V_i on the elements of this thread; h in shared memory
__device__ __forceinline__ void subtract(const cplx* V, long long ldv, int nv, const cplx* hs,
                                         cplx* w, long long n) {
  for (long long e = blockIdx.x * (long long)AT + threadIdx.x; e < n; e += (long long)gridDim.x * AT) {
    cplx acc = w[e];
    for (int i = 0; i < nv; ++i) cfma(acc, hs[i], V[(long long)i * ldv + e]);
    w[e] = acc;
  }
}

// True in the block that arrives last, which then sees what the others wrote
// before they arrived; leaves the counter at zero.
__device__ __forceinline__ bool last_block(unsigned int* counter) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
    if (last) *counter = 0u;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// The block's shares to `partial` (2 nv doubles per block), and in the last block
// the sums, in block order, to out
__device__ __forceinline__ void finish_dots(int nv, double (*sh)[2 * MAXV + 6], cplx* partial,
                                            cplx* out, unsigned int* counter) {
  __syncthreads();
  double* p = reinterpret_cast<double*>(partial);
  for (int c = threadIdx.x; c < 2 * nv; c += AT) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < AW; ++w) t += sh[w][c];
    p[(long long)blockIdx.x * 2 * nv + c] = t;
  }
  if (!last_block(counter)) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int i = wid; i < nv; i += AW) {
    double sr = 0.0, si = 0.0;
    for (unsigned int b = lane; b < gridDim.x; b += 32) {
      const cplx v = __ldcg(partial + (long long)b * nv + i);
      sr += v.x;
      si += v.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sr += __shfl_xor_sync(0xffffffffu, sr, o);
      si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    if (lane == 0) out[i] = cmake(sr, si);
  }
}

// Two real sums over the block (valid in thread 0)
__device__ __forceinline__ void block_sum_pair(double& a, double& b) {
  __shared__ double sh[AW][2];
  a = warp_sum(a);
  b = warp_sum(b);
  if ((threadIdx.x & 31) == 0) {
    sh[threadIdx.x >> 5][0] = a;
    sh[threadIdx.x >> 5][1] = b;
  }
  __syncthreads();
  a = b = 0.0;
#pragma unroll
  for (int w = 0; w < AW; ++w) {
    a += sh[w][0];
    b += sh[w][1];
  }
}

// Sums over all blocks' (a, b) in the last block, in every lane of its first
// warp; returns false in all other threads
__device__ __forceinline__ bool total_pair(double& a, double& b, cplx* partial,
                                           unsigned int* counter) {
  if (threadIdx.x == 0) partial[blockIdx.x] = cmake(a, b);
  if (!last_block(counter) || threadIdx.x >= 32) return false;
  a = b = 0.0;
  for (unsigned int k = threadIdx.x; k < gridDim.x; k += 32) {
    const cplx v = __ldcg(partial + k);
    a += v.x;
    b += v.y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  return true;
}

__device__ __forceinline__ cplx& Hc(GmresState* s, int i, int j) { return s->H[j * (32 + 1) + i]; }

// r = B - r, |r|^2 and |B|^2, and the start of the cycle
__global__ void __launch_bounds__(AT)
k_arnoldi_start(cplx* r, const cplx* B, long long n, GmresState* s, cplx* partial,
                unsigned int* counter) {
  double a = 0.0, b = 0.0;
  for (long long e = blockIdx.x * (long long)AT + threadIdx.x; e < n; e += (long long)gridDim.x * AT) {
    const cplx be = B[e], v = csub(be, r[e]);
    r[e] = v;
    a = fma(v.x, v.x, fma(v.y, v.y, a));
    b = fma(be.x, be.x, fma(be.y, be.y, b));
  }
  block_sum_pair(a, b);
  if (!total_pair(a, b, partial, counter)) return;
  const int lane = threadIdx.x;
  for (int i = lane; i < 33; i += 32) s->g[i] = cmake(0.0, 0.0);
  s->y[lane] = cmake(0.0, 0.0);
  for (int i = lane; i < 33 * 32; i += 32) s->H[i] = cmake(0.0, 0.0);
  __syncwarp();
  if (lane != 0) return;
  const double beta = sqrt(a);
  s->beta = beta;
  s->bnorm = sqrt(b);
  s->steps = 0;
  s->breakdown = 0;
  s->res = beta;
  if (beta > 0.0 && isfinite(beta)) {
    s->active = 1;
    s->inv_h = 1.0 / beta;
    s->g[0] = cmake(beta, 0.0);
  } else {
    s->active = 0;
    s->inv_h = 0.0;
  }
}

__global__ void __launch_bounds__(AT)
k_arnoldi_dot(const cplx* V, long long ldv, int nv, const cplx* w, long long n, GmresState* s,
              cplx* partial, unsigned int* counter) {
  if (s->active == 0) return;
  __shared__ double sh[AW][2 * MAXV + 6];
  dot_shares(V, ldv, nv, w, n, sh);
  finish_dots(nv, sh, partial, s->h, counter);
}

__global__ void __launch_bounds__(AT)
k_arnoldi_mid(const cplx* V, long long ldv, int nv, cplx* w, long long n, GmresState* s,
              cplx* partial, unsigned int* counter) {
  if (s->active == 0) return;
  __shared__ double sh[AW][2 * MAXV + 6];
  __shared__ cplx hs[MAXV];
  for (int i = threadIdx.x; i < nv; i += AT) hs[i] = cscale(s->h[i], -1.0);
  __syncthreads();
  subtract(V, ldv, nv, hs, w, n);
  dot_shares(V, ldv, nv, w, n, sh);
  finish_dots(nv, sh, partial, s->h + 32, counter);
}

// Column j of H from the two passes' projections and |w|^2, the Givens update
// and the tests that end the cycle (one warp: the column and the earlier
// rotations are fetched together, the chain of rotations runs in lane 0).
__device__ void gmres_step(GmresState* s, int j, int m, double brel, double ltol, double wnorm2,
                           cplx* col, cplx* cs, cplx* sn) {
  const int lane = threadIdx.x;
  double c2 = 0.0;
  if (lane <= j) {
    const cplx h = cadd(s->h[lane], s->h[32 + lane]);
    col[lane] = h;
    c2 = fma(h.x, h.x, h.y * h.y);
    if (lane < j) {
      cs[lane] = s->cs[lane];
      sn[lane] = s->sn[lane];
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c2 += __shfl_xor_sync(0xffffffffu, c2, o);
  __syncwarp();
  if (lane == 0) {
    s->wnorm2 = wnorm2;
    const double hj1 = sqrt(wnorm2);
    // |A v_j|^2 = sum_i |h_ij|^2 + h_{j+1,j}^2 (Arnoldi relation); a happy
    // breakdown is a new direction that is negligible against it
    const double col2 = wnorm2 + c2;
    cplx a = col[0];
    for (int i = 0; i < j; ++i) {
      const cplx b = col[i + 1], c = cs[i], t = sn[i];
      col[i] = cadd(cmul(c, a), cmul(t, b));
      a = csub(cmul(c, b), cmul(cconj(t), a));
    }
    // new rotation zeroing h_{j+1,j}
    const double an = hypot(a.x, a.y);
    const double r = hypot(an, hj1);
    cplx c, t;
    if (r == 0.0) {
      c = cmake(1.0, 0.0); t = cmake(0.0, 0.0);
    } else if (an == 0.0) {
      c = cmake(0.0, 0.0); t = cmake(1.0, 0.0);
    } else {
      c = cmake(an / r, 0.0);
      t = cscale(a, hj1 / (an * r));
    }
    s->cs[j] = c;
    s->sn[j] = t;
    col[j] = (an == 0.0) ? cmake(hj1, 0.0) : cscale(a, r / an);
    const cplx gj = s->g[j];
    const cplx g1 = cscale(cmul(cconj(t), gj), -1.0);
    s->g[j] = cmul(c, gj);
    s->g[j + 1] = g1;
    const double res = hypot(g1.x, g1.y);
    s->res = res;
    s->steps = j + 1;
    if (!(hj1 > brel * sqrt(col2)) || !isfinite(hj1)) {
      s->breakdown = 1;
      s->active = 0;
    } else if (ltol > 0.0 && res <= ltol * s->bnorm) {
      s->active = 0;
    } else if (j + 1 >= m) {
      s->active = 0;
    } else {
      s->inv_h = 1.0 / hj1;
    }
  }
  __syncwarp();
  if (lane <= j) Hc(s, lane, j) = col[lane];
}

__global__ void __launch_bounds__(AT)
k_arnoldi_end(const cplx* V, long long ldv, int j, int m, cplx* w, long long n, double brel,
              double ltol, GmresState* s, cplx* partial, unsigned int* counter) {
  if (s->active == 0) return;
  __shared__ cplx hs[MAXV], cs[MAXV], sn[MAXV];
  for (int i = threadIdx.x; i <= j; i += AT) hs[i] = cscale(s->h[32 + i], -1.0);
  __syncthreads();
  double a = 0.0, b = 0.0;
  for (long long e = blockIdx.x * (long long)AT + threadIdx.x; e < n; e += (long long)gridDim.x * AT) {
    cplx acc = w[e];
    for (int i = 0; i <= j; ++i) cfma(acc, hs[i], V[(long long)i * ldv + e]);
    w[e] = acc;
    a = fma(acc.x, acc.x, fma(acc.y, acc.y, a));
  }
  block_sum_pair(a, b);
  if (!total_pair(a, b, partial, counter)) return;
  gmres_step(s, j, m, brel, ltol, a, hs, cs, sn);
}

// y of the triangular system (one warp; row i's products by the lanes)
__global__ void __launch_bounds__(32) k_gmres_finish(GmresState* s) {
  __shared__ cplx y[MAXV];
  const int k = s->steps, lane = threadIdx.x;
  for (int i = k - 1; i >= 0; --i) {
    const int l = i + 1 + lane;
    double sr = 0.0, si = 0.0;
    if (l < k) {
      const cplx t = cmul(Hc(s, i, l), y[l]);
      sr = t.x;
      si = t.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sr += __shfl_xor_sync(0xffffffffu, sr, o);
      si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    if (lane == 0) {
      const cplx acc = csub(s->g[i], cmake(sr, si)), d = Hc(s, i, i);
      const double dn = d.x * d.x + d.y * d.y;
      const cplx v = (dn > 0.0) ? cscale(cmul(acc, cconj(d)), 1.0 / dn) : cmake(0.0, 0.0);
      y[i] = v;
      s->y[i] = v;
    }
    __syncwarp();
  }
}

}  // namespace

cudaError_t vec_copy(cplx* y, const cplx* x, long long n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  count_launches(1);
  k_copy<<<grid_for(n), VT, 0, st>>>(y, x, n);
  return cudaGetLastError();
}
cudaError_t vec_zero(cplx* y, long long n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  count_launches(1);
  k_zero<<<grid_for(n), VT, 0, st>>>(y, n);
  return cudaGetLastError();
}
cudaError_t vec_axpby(cplx* y, const cplx* x, cplx a, cplx b, long long n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  count_launches(1);
  k_axpby<<<grid_for(n), VT, 0, st>>>(y, x, a, b, n);
  return cudaGetLastError();
}
cudaError_t vec_block_axpy(const cplx* V, long long ldv, int nv, const int* nv_dev,
                           const cplx* h, double sign, cplx* w, long long n, const int* active,
                           cudaStream_t st) {
  if (nv <= 0 || n <= 0) return cudaSuccess;
  if (nv > MAXV) return cudaErrorInvalidValue;
  count_launches(1);
  k_block_axpy<<<grid_for(n), VT, 0, st>>>(V, ldv, nv, nv_dev, h, sign, w, n, active);
  return cudaGetLastError();
}
cudaError_t vec_norm2(const cplx* x, long long n, double* out, double* partial,
                      const int* active, cudaStream_t st) {
  const int g = grid_for(n);
  count_launches(1);
  k_norm2_partial<<<g, VT, 0, st>>>(x, n, partial, active);
  count_launches(1);
  k_reduce_real<<<1, 32, 0, st>>>(partial, g, out, active);
  return cudaGetLastError();
}
namespace {
__global__ void k_scale_scalar(double* v, double s) {
  if (threadIdx.x == 0) *v *= s;
}
}  // namespace

cudaError_t scaled_norm2(const cplx* x, long long n, double scale, double* out, double* partial,
                         cudaStream_t st) {
  cudaError_t e = vec_norm2(x, n, out, partial, nullptr, st);
  if (e != cudaSuccess) return e;
  count_launches(1);
  k_scale_scalar<<<1, 32, 0, st>>>(out, scale);
  return cudaGetLastError();
}

cudaError_t vec_scale_dev(cplx* y, const double* scale, long long n, const int* active,
                          cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  count_launches(1);
  k_scale_dev<<<grid_for(n), VT, 0, st>>>(y, scale, n, active);
  return cudaGetLastError();
}
cudaError_t env_trace(const cplx* L, const cplx* R, int D, int m, int n, cplx* out,
                      cplx* partial, cudaStream_t st) {
  const long long tot = (long long)D * m * n;
  const int g = grid_for(tot);
  count_launches(1);
  k_env_trace<<<g, VT, 0, st>>>(L, R, D, m, n, partial);
  count_launches(1);
  k_reduce_cplx<<<1, 32, 0, st>>>(partial, g, 1, out, nullptr);
  return cudaGetLastError();
}
cudaError_t apply_site_op(const cplx* O, const cplx* K, cplx* Kout, int chl, int d, int chr,
                          cudaStream_t st) {
  const long long tot = (long long)chl * d * chr;
  if (tot <= 0) return cudaSuccess;
  count_launches(1);
  k_site_op<<<grid_for(tot), VT, 0, st>>>(O, K, Kout, chl, d, chr);
  return cudaGetLastError();
}
cudaError_t mix_apply(const MixPlan& plan, const MixStrides& s, int P, int Q, const cplx* in,
                      long long iP, long long iQ, cplx* out, long long oP, long long oQ,
                      cudaStream_t st) {
  if (plan.nrows > MIX_MAX || plan.ncols > MIX_MAX) return cudaErrorInvalidValue;
  const long long tot = (long long)P * Q;
  if (tot <= 0) return cudaSuccess;
  long long g = (long long)P * ((Q + MIX_Q - 1) / MIX_Q);
  if (g > 152 * 8) g = 152 * 8;
  count_launches(1);
  k_mix<<<(int)g, MIX_Q * MIX_G, 0, st>>>(plan, s, P, Q, in, iP, iQ, out, oP, oQ);
  return cudaGetLastError();
}
cudaError_t arnoldi_start(cplx* r, const cplx* B, long long n, GmresState* s, cplx* partial,
                          unsigned int* counter, cudaStream_t st) {
  count_launches(1);
  k_arnoldi_start<<<arnoldi_grid(n), AT, 0, st>>>(r, B, n, s, partial, counter);
  return cudaGetLastError();
}
cudaError_t arnoldi_step(const cplx* V, long long ldv, int j, int m, cplx* w, long long n,
                         double breakdown_rel, double local_tol, GmresState* s, cplx* partial,
                         unsigned int* counter, cudaStream_t st) {
  if (j < 0 || j >= MAXV || n <= 0) return cudaErrorInvalidValue;
  const int g = arnoldi_grid(n);
  count_launches(3);
  k_arnoldi_dot<<<g, AT, 0, st>>>(V, ldv, j + 1, w, n, s, partial, counter);
  k_arnoldi_mid<<<g, AT, 0, st>>>(V, ldv, j + 1, w, n, s, partial, counter);
  k_arnoldi_end<<<g, AT, 0, st>>>(V, ldv, j, m, w, n, breakdown_rel, local_tol, s, partial, counter);
  return cudaGetLastError();
}
cudaError_t gmres_finish(GmresState* s, cudaStream_t st) {
  count_launches(1);
  k_gmres_finish<<<1, 32, 0, st>>>(s);
  return cudaGetLastError();
}

}  // namespace ite
