// Preconditioner of the one-sided Jacobi of the truncated splits.
//
// The FP64 Jacobi (svd.cu) is a chain of one grid barrier per round and of
// FP64 work on a pipe that issues two DFMA per clock and SM: 512 rows take 11
// sweeps of 511 rounds of about 10 us.  Nearly all of that work only brings
// rows that start far from orthogonal to a few digits of orthogonality, which
// does not need FP64.  So the split first rotates the rows of R (k x p) by a
// unitary V found in fp32, V R with rows orthogonal to about 1e-6:
//   1. k_jacobi32: one-sided block Jacobi in fp32 on the rows of [R | I], one
//      block pair (32 rows) per thread-block cluster and step, whose Gram
//      matrix is diagonalised by Jacobi rotations in shared memory;
//   2. V is made unitary to FP64 rounding by two or three Newton-Schulz steps
//      V <- V - (V V^H - I) V / 2, and applied, S = V R, in FP64 (FP64-class)
//      GEMMs: S^H S = R^H R to rounding, whatever the quality of V;
//   3. twice, the Gram matrix G = S S^H gives the first-order rotations
//      E_ij = t e^{i theta} of every pair that is not yet orthogonal (the
//      Jacobi rotation's tangent, kept only where it is small), and
//      S <- S + (E + E^2/2 - E^4/8) S, unitary to E^6: quadratic convergence
//      for well separated rows;
//   4. a last Gram matrix lists the rows that still have a pair above the
//      Jacobi's tolerance (members of near-degenerate groups, or all rows if
//      a check below failed); the FP64 Jacobi runs on those rows only.
// Every transformation applied is unitary to FP64 rounding, and the FP64
// Jacobi's criterion decides what remains.  Rows of very different weight: an
// FP64-class product is accurate relative to the largest entry of a row of its
// left and of a column of its right factor, so V R and D S alone would leave the
// light rows an error of 2^-56 of the heaviest (a singular value of 1e-10 of the
// largest was off by 3e-8 of itself, for 300 rows graded along the columns).  The
// rows of R and S are therefore divided by the powers of two next to their norms,
// and the columns of V and D multiplied by them (rexp, exact, while the operands are
// cut): the entries of (V diag d)_i are then what the terms of row i weigh, and the
// singular values keep the relative accuracy of FP64 products (1e-15 in that case).
// S is updated by small corrections D S rather than replaced by Q S.
// Guards: V is dropped (S = R, all rows go to the Jacobi) unless no bounded wait ran
// out in k_jacobi32 and |V V^H - I|_inf < 1e-2, from which three Newton-Schulz steps
// reach rounding; a correction is dropped unless |E|_inf <= 2e-3.  What a guard drops
// costs time, not the result: the FP64 Jacobi takes the rows that are left.
#include <cooperative_groups.h>

#include <atomic>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace ite {
namespace {

// control words (PreCtl in device memory, cleared before each use)
constexpr int C_ARRIVE = 0, C_ERR = 4, C_SWEEPS = 5;
constexpr int C_OK = 8, C_GE = 9, C_GW = 10, C_GW2 = 11, C_COUNT = 12, C_GN = 13;
constexpr int C_DELTA = 16, C_NU = 18;        // 64-bit words
constexpr int C_OFF = 24;                     // per-sweep largest overlap (float bits)
constexpr int C_WORDS = 64;
constexpr int kSweeps32 = 16;
static_assert(C_OFF + kSweeps32 <= C_WORDS, "control words");

constexpr int PB = 16;                        // rows of a block
constexpr int PM = 2 * PB;                    // rows of a block pair
constexpr int PT = 256;                       // threads per CTA
constexpr int GLD = PM + 1;                   // padded row of the Gram matrix
constexpr int QLD = PM + 2;                   // padded row of Q^T (16-byte aligned pairs)
constexpr float kStop32 = 1e-3f;              // largest overlap of the last sweep (its square remains)
constexpr float kRot32 = 2e-7f;               // overlaps below this are fp32 rounding
constexpr float kTiny32 = 1e-34f;             // squared norms below this (of 1) are left alone

struct Pre32 {
  float2* R;                                  // kp rows of pl, the scaled rows of R
  float2* V;                                  // kp rows of vl, the accumulated rotation
  int k, kp, pl, vl, nb;                      // rows, padded rows, row strides, blocks
  int pc, vc, chunk;                          // columns of R and V per CTA, columns staged at once
  unsigned int* ver;                          // (block, CTA of a cluster): steps done
};

// Barrier over the clusters' first CTAs: arrivals are counted up without a reset,
// barrier number t is passed at t n of them (one trip to L2 to arrive, one to
// see it).  Bounded: after 2^24 polls the error flag is set, and a wait also
// gives up as soon as another has set it.
__device__ bool leader_barrier(unsigned int* st, unsigned int target) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(st + C_ARRIVE) : "memory");
  unsigned long long spins = 0;
  for (;;) {
    unsigned int seen;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(st + C_ARRIVE) : "memory");
    if ((int)(seen - target) >= 0) return true;
    if (*((volatile unsigned int*)(st + C_ERR)) != 0u) return false;
    if (++spins > (1ull << 24)) {
      atomicExch(st + C_ERR, 1u);
      return false;
    }
  }
}

__device__ __forceinline__ int seat(int pos, int round, int n) {
  return pos == 0 ? 0 : ((pos - 1 + round) % (n - 1)) + 1;
}

// Local column c of this CTA in the concatenated row [R | V] (aligned pairs of
// columns: pc and vc are multiples of 4).
__device__ __forceinline__ float4* col_ptr(const Pre32& a, int row, int rank, int c) {
  float2* p = c < a.pc ? a.R + (long long)row * a.pl + (long long)rank * a.pc + c
                       : a.V + (long long)row * a.vl + (long long)rank * a.vc + (c - a.pc);
  return reinterpret_cast<float4*>(p);
}

__device__ __forceinline__ void copy16(float2* dst, const float4* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (unsigned int)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}

__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Rotation x' = c x - s y, y' = conj(s) x + c y of two rows with squared norms
// al, be and inner product g = x y^H that makes them orthogonal; returns what it
// moves from al to be.  Written in the overlap h = g / (|x| |y|) and the ratio of
// the norms, which stay in range for rows of any weight: with zeta = (be - al) /
// (2 |g|) and r = 1 / sqrt(1 + zeta^2), cos 2a = |zeta| r and sin 2a = r, so
// c^2 = (1 + |zeta| r) / 2 and |s| = r / (2 c).  Every round waits for this chain:
// four dependent approximate inverse square roots (2^-22.9 relative) and no branch;
// the last two take one Newton-Raphson step, y (3 - x y^2) / 2, because their errors
// would stand in c^2 + |s|^2 - 1.  Error bounds, from those of the approximations (the
// kernel below gives the values): c 2^-21, s 2^-19 relative, c^2 + |s|^2 - 1 2^-21.
__device__ __forceinline__ float rotation(float al, float be, float2 g, float& c, float& sx,
                                          float& sy, float& off) {
  const bool rows = al > kTiny32 && be > kTiny32;
  const float ra = rsqrt_approx(rows ? al : 1.f), rb = rsqrt_approx(rows ? be : 1.f);
  const float rab = ra * rb, hx = g.x * rab, hy = g.y * rab;
  const float h2 = fmaf(hx, hx, hy * hy);
  const bool on = rows && h2 > kRot32 * kRot32;
  const float ih = rsqrt_approx(on ? h2 : 1.f);
  const float df = be - al;
  const float z = 0.5f * fabsf(df) * rab * ih;
  // r = 1 / z where 1 + z^2 is z^2 (and may be infinite): s has to stay exact, it
  // multiplies a row that can be 1e17 times as long as the other
  const bool far = z > 1e9f;
  const float w = fmaf(z, z, 1.f), rf = rcp_approx(z);
  float r = rsqrt_approx(w);
  r = far ? rf : r * fmaf(-0.5f * w * r, r, 1.5f);
  const float c2 = far ? 1.f : fmaf(0.5f * z, r, 0.5f);
  float q = rsqrt_approx(c2);
  q = q * fmaf(-0.5f * c2 * q, q, 1.5f);      // 1 / c
  const float sn = on ? copysignf(0.5f * r * q * ih, df) : 0.f;
  c = on ? c2 * q : 1.f;
  sx = sn * hx;
  sy = sn * hy;
  off = fmaxf(off, on ? h2 * ih : 0.f);
  // t |g| = (|s| / c) |h| |x| |y|
  return sn * q * h2 * (al * ra) * (be * rb);
}

// The rotation of n pairs, for its test.
__global__ void k_rotations(int n, const float* al, const float* be, const float2* g, float* c,
                            float2* s) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    float off = 0.f;
    rotation(al[i], be[i], g[i], c[i], s[i].x, s[i].y, off);
  }
}

// Columns of one rank of a block have been through `step` steps: each CTA needs
// nothing but its own columns of the two blocks, so it waits for the CTAs that
// wrote these instead of for all.  Bounded; after a failed wait anywhere the
// sweep is run out without waiting (its result is discarded).
__device__ __forceinline__ void wait_block(const unsigned int* ver, unsigned int step,
                                           unsigned int* st) {
  for (unsigned int spins = 0;; ++spins) {
    unsigned int seen;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(ver) : "memory");
    if ((int)(seen - step) >= 0) return;
    if ((spins & 63u) == 63u && *((volatile unsigned int*)(st + C_ERR)) != 0u) return;
    if (spins > (1u << 24)) {
      atomicExch(st + C_ERR, 1u);
      return;
    }
  }
}

__device__ __forceinline__ void publish_block(unsigned int* ver, unsigned int step) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(ver), "r"(step) : "memory");
}

__device__ __forceinline__ float2 conj(const float2& a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 neg(const float2& a) { return make_float2(-a.x, -a.y); }

// c x + f y in this order of operations wherever it stands.
__device__ __forceinline__ float2 turn(float c, const float2& x, const float2& f, const float2& y) {
  return make_float2(fmaf(c, x.x, fmaf(f.x, y.x, -__fmul_rn(f.y, y.y))),
                     fmaf(c, x.y, fmaf(f.x, y.y, __fmul_rn(f.y, y.x))));
}

// Where the entries of round r + 1's pair t stand before round r has turned them:
// pair (m, n = m ^ (r + 1)), the partners m_ = m ^ r, n_ = n ^ r of round r, the
// pairs pm, pn of round r that m and n are in, and 1 or -1 as they are the second
// or the first there.  m and n are exchanged (swap) where that puts the lower pair
// first, as in the update's blocks.
struct Ahead {
  int mn, mn_, m_n, m_n_, mm, nn, pm, pn;
  float sm, sn;
  bool swap;
  __device__ __forceinline__ Ahead(int r, int t) {
    const int r2 = min(r + 1, PM - 1);
    const int hb = 31 - __clz(r), low = (1 << hb) - 1, low2 = (1 << (31 - __clz(r2))) - 1;
    int m = ((t & ~low2) << 1) | (t & low2), n = m ^ r2;
    auto index = [&](int x) {
      const int f = (x >> hb) & 1 ? x ^ r : x;
      return ((f >> 1) & ~low) | (f & low);
    };
    pm = index(m);
    pn = index(n);
    swap = pm > pn;
    if (swap) {
      int x = m;
      m = n;
      n = x;
      x = pm;
      pm = pn;
      pn = x;
    }
    mn = m * GLD + n;
    mn_ = m * GLD + (n ^ r);
    m_n = (m ^ r) * GLD + n;
    m_n_ = (m ^ r) * GLD + (n ^ r);
    mm = m * (GLD + 1);
    nn = n * (GLD + 1);
    sm = (m >> hb) & 1 ? 1.f : -1.f;
    sn = (n >> hb) & 1 ? 1.f : -1.f;
  }
};

// Rows m, n of N columns of Q, STEP apart, turned by the rotation A = (c, s).
template <int N, int STEP>
__device__ __forceinline__ void turn_q(float2* q, int m, int n, const float4& A) {
  const float2 sn = make_float2(A.y, A.z);
  float2 x[N], y[N];
#pragma unroll
  for (int h = 0; h < N; ++h) {
    x[h] = q[h * STEP * QLD + m];
    y[h] = q[h * STEP * QLD + n];
  }
#pragma unroll
  for (int h = 0; h < N; ++h) {
    q[h * STEP * QLD + m] = turn(A.x, x[h], neg(sn), y[h]);
    q[h * STEP * QLD + n] = turn(A.x, y[h], conj(sn), x[h]);
  }
}

// Rows r0..r0+7 of Q S for NC columns per lane, written to their sorted places.
template <int NC>
__device__ __forceinline__ void apply_rows(const Pre32& a, const float2* S, const float2* QT,
                                           const int* pos, int ld, int cb, int n, int r0, int u,
                                           int v, int rank, int c0) {
  const int lane = threadIdx.x & 31, half = threadIdx.x >> 7;
  const int c = cb + 32 * half + lane;
  const float2* sp[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) sp[j] = S + (c + 64 * j < n ? c + 64 * j : 0);
  float2 o[8][NC];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < NC; ++j) o[i][j] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int m = 0; m < PM; ++m) {
    float2 s[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) s[j] = sp[j][m * ld];
    const float4* qp = reinterpret_cast<const float4*>(QT + m * QLD + r0);
#pragma unroll
    for (int i2 = 0; i2 < 4; ++i2) {
      const float4 q = qp[i2];
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        float2& o0 = o[2 * i2][j];
        float2& o1 = o[2 * i2 + 1][j];
        o0.x = fmaf(q.x, s[j].x, fmaf(-q.y, s[j].y, o0.x));
        o0.y = fmaf(q.x, s[j].y, fmaf(q.y, s[j].x, o0.y));
        o1.x = fmaf(q.z, s[j].x, fmaf(-q.w, s[j].y, o1.x));
        o1.y = fmaf(q.z, s[j].y, fmaf(q.w, s[j].x, o1.y));
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int at = pos[r0 + i];
    const int row = at < PB ? u * PB + at : v * PB + at - PB;
#pragma unroll
    for (int j = 0; j < NC; ++j)
      if (c + 64 * j < n) *reinterpret_cast<float2*>(col_ptr(a, row, rank, c0 + c + 64 * j)) = o[i][j];
  }
}

// One cluster per block pair, the columns of the pair's rows dealt to its
// CTAs.  Per step: each CTA stages its columns, forms its share of the 32 x 32
// Gram matrix, the shares are added through distributed shared memory in a
// fixed order, every CTA diagonalises the sum the same way and applies the
// result to its own columns.
// Bound: latency and shared memory.  Clocks per step at k = 512 (16 pairs, 6 CTAs
// each, 31 steps a sweep): wait for the blocks 1.7k, copy in 1.7k, Gram 4.3k, sum
// 3.3k, the 16 or 31 dependent rounds 13.8k (620 each: the chain of approximate
// square roots on warp 4), rows 11k; 19 us in all.  With a barrier over the grid
// after every step, the rotations formed before the update and 2 x 2 tiles in the
// Gram matrix: 23.7 us.  16-row blocks: 8-row ones need twice the steps for the
// same number of rounds, 32-row ones leave half the SMs without a pair.  Whole
// 512 x 512 split (chi_max 256, cutoff 1e-10): 69 ms with the FP64 Jacobi alone,
// 9.0 ms with the preconditioner (no FP64 sweep is left); 1024 x 1024: 325 and 35.
__global__ void __launch_bounds__(PT, 1)
k_jacobi32(Pre32 a, unsigned int* st) {
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int ncl = gridDim.x / C, cid = blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  extern __shared__ float4 dyn[];
  float2* parts = reinterpret_cast<float2*>(dyn);           // PM x GLD, by parity of the pair
  float2* G = parts + 2 * PM * GLD;                         // PM x GLD
  float2* G2 = G + PM * GLD;                                // PM x GLD
  float2* QT = G2 + PM * GLD;                               // PM x QLD: QT[c][r] = Q[r][c]
  float2* S = QT + PM * QLD;                                // PM x ld
  __shared__ int s_pos[PM];
  __shared__ int s_off, s_ok;
  __shared__ float4 s_rot[2][PB];             // rotations (c, s, t |g|) of a round, by its parity
  const int lc = a.pc + a.vc, ld = a.chunk + 2;
  const bool resident = lc <= a.chunk;
  const int tx = tid & 15;
  const int gk = tid >> 6, gi = (tid >> 3) & 7, gj = tid & 7;      // of the Gram matrix
  unsigned int passed = 0;                    // barrier arrivals so far
  // the two row pairs pa < pb whose block of G this thread turns (tid < 120):
  // rows x and 15 - x of the 16 x 16 triangle make one row of 15 blocks
  const int fx = min(tid, 119) / 15, fy = min(tid, 119) - 15 * fx;
  const int pa = fy >= fx ? fx : 15 - fx, pb = fy >= fx ? fy + 1 : 16 - fx + fy;

  // rows of the pair (u, v): 0..15 of block u, then 0..15 of block v; each warp
  // copies four rows
  auto stage = [&](int u, int v, int c0, int n) {
    const int r0 = 4 * warp;
    const int row = (r0 < PB ? u * PB : (v - 1) * PB) + r0;
    for (int c = 2 * lane; c < n; c += 64)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        copy16(S + (r0 + i) * ld + c, col_ptr(a, row + i, rank, c0 + c));
    asm volatile("cp.async.wait_all;" ::: "memory");
  };

  int pairs_done = 0;
  for (int sw = 0; sw < kSweeps32; ++sw) {
    for (int rd = 0; rd < a.nb - 1; ++rd) {
      const unsigned int step = (unsigned int)(sw * (a.nb - 1) + rd);
      for (int k = cid; k < a.nb / 2; k += ncl, ++pairs_done) {
        int u = seat(k, rd, a.nb), v = seat(a.nb - 1 - k, rd, a.nb);
        if (u > v) { const int t = u; u = v; v = t; }
        // this CTA's columns of the two blocks, as the last step left them
        if (tid == 0) {
          wait_block(a.ver + u * 8 + rank, step, st);
          wait_block(a.ver + v * 8 + rank, step, st);
        }
        __syncthreads();
        float2* const part = parts + (pairs_done & 1) * PM * GLD;
        // ---- share of the Gram matrix: four groups of 64 threads take every
        // fourth pair of columns, thread (gi, gj) of a group the rows gi + 8 x by
        // gj + 8 y, x <= y (the others are mirror images)
        float2 acc[10];
#pragma unroll
        for (int i = 0; i < 10; ++i) acc[i] = make_float2(0.f, 0.f);
        for (int c0 = 0; c0 < (resident ? 1 : a.pc); c0 += a.chunk) {
          const int n = resident ? lc : min(a.chunk, a.pc - c0);
          const int ng = resident ? a.pc : n;
          stage(u, v, c0, n);
          __syncthreads();
          for (int c = 2 * gk; c < ng; c += 8) {
            float4 x[4], y[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              x[i] = *reinterpret_cast<const float4*>(S + (gi + 8 * i) * ld + c);
              y[i] = *reinterpret_cast<const float4*>(S + (gj + 8 * i) * ld + c);
            }
            int e = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = i; j < 4; ++j, ++e) {
                // x conj(y)
                acc[e].x = fmaf(x[i].x, y[j].x, fmaf(x[i].y, y[j].y, acc[e].x));
                acc[e].y = fmaf(x[i].y, y[j].x, fmaf(-x[i].x, y[j].y, acc[e].y));
                acc[e].x = fmaf(x[i].z, y[j].z, fmaf(x[i].w, y[j].w, acc[e].x));
                acc[e].y = fmaf(x[i].w, y[j].z, fmaf(-x[i].z, y[j].w, acc[e].y));
              }
          }
          if (!resident) __syncthreads();
        }
        // groups 1-3 hand theirs to group 0 (G, G2 and QT are free here)
        float2* const mine = gk == 0 ? part : gk == 1 ? G : gk == 2 ? G2 : QT;
        if (gk > 0) {
          int e = 0;
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = i; j < 4; ++j, ++e) mine[(gi + 8 * i) * GLD + gj + 8 * j] = acc[e];
        }
        __syncthreads();
        if (gk == 0) {
          int e = 0;
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = i; j < 4; ++j, ++e) {
              const int at = (gi + 8 * i) * GLD + gj + 8 * j;
              const float2 p = G[at], q = G2[at], r = QT[at];
              part[at] = make_float2((acc[e].x + p.x) + (q.x + r.x), (acc[e].y + p.y) + (q.y + r.y));
            }
        }
        cl.sync();
        // ---- sum of the shares (upper triangle, mirrored); Q = I
        for (int e = tid; e < PM * (PM + 1) / 2; e += PT) {
          // rows x and 31 - x of the triangle make one row of 33 entries
          const int x = e / (PM + 1), y = e - x * (PM + 1);
          const int i = y > x ? x : PM - 1 - x, j = y > x ? y - 1 : PM - 1 - y;
          float2 t[8];
#pragma unroll
          for (int r = 0; r < 8; ++r)
            t[r] = r < C ? cl.map_shared_rank(part, r)[i * GLD + j] : make_float2(0.f, 0.f);
          float2 s = t[0];
#pragma unroll
          for (int r = 1; r < 8; ++r) {
            s.x += t[r].x;
            s.y += t[r].y;
          }
          if (i == j) {
            // padding rows sort last and never rotate
            const int row = i < PB ? u * PB + i : v * PB + i - PB;
            G[i * GLD + i] = make_float2(row < a.k ? s.x : -1.f, 0.f);
          } else {
            G[i * GLD + j] = s;
            G[j * GLD + i] = make_float2(s.x, -s.y);
          }
        }
        for (int e = tid; e < PM * PM; e += PT)
          QT[(e >> 5) * QLD + (e & 31)] = make_float2((e >> 5) == (e & 31) ? 1.f : 0.f, 0.f);
        if (tid == 0) s_off = 0;
        __syncthreads();
        // ---- one cyclic sweep of rotations, all pairs of the 32 rows in every
        // fourth step, only those across the two blocks (16 rounds instead of
        // 31) in the others: as many sweeps as with all pairs every time.
        // Round r pairs row i with row i ^ r; pair t is the t-th i whose highest
        // bit of r is clear.  Warps 0-3 turn the 120 blocks of two different pairs
        // from one copy of G to the other (upper block, mirrored), warps 5-7 the
        // pairs' own blocks and half of Q (warps 0-3 the other half).  Warp 4
        // meanwhile turns just the entries that the next round's pairs need and
        // forms their rotations, so that the chain of square roots runs beside the
        // update, not before it: 620 clocks a round, 850 one after the other.
        float off = 0.f;
        float2 *Ga = G, *Gb = G2;
        const int rfirst = (rd & 3) == 0 ? 1 : PB;
        if (warp == 4) {
          const int hb = 31 - __clz(rfirst), low = (1 << hb) - 1;
          const int m = ((tx & ~low) << 1) | (tx & low), n = m ^ rfirst;
          float4 q;
          q.w = rotation(Ga[m * GLD + m].x, Ga[n * GLD + n].x, Ga[m * GLD + n], q.x, q.y, q.z, off);
          if (lane < PB) s_rot[rfirst & 1][tx] = q;
        }
        Ahead ahead(rfirst, tx);
        __syncthreads();
        for (int r = rfirst; r < PM; ++r) {
          const int hb = 31 - __clz(r), low = (1 << hb) - 1;
          auto first = [&](int t) { return ((t & ~low) << 1) | (t & low); };
          const float4* const rot = s_rot[r & 1];
          if (warp < 4) {
            const int mq = first(tx);
            turn_q<2, 8>(QT + (16 + (tid >> 4)) * QLD, mq, mq ^ r, rot[tx]);
            if (tid < 120) {
              const int i = first(pa), j = i ^ r, k2 = first(pb), l2 = k2 ^ r;
              const float4 A = rot[pa], B = rot[pb];
              const float2 b00 = Ga[i * GLD + k2], b01 = Ga[i * GLD + l2];
              const float2 b10 = Ga[j * GLD + k2], b11 = Ga[j * GLD + l2];
              const float2 sa = make_float2(A.y, A.z), sb = make_float2(B.y, B.z);
              // rows: x' = c x - s y, y' = conj(s) x + c y
              const float2 p00 = turn(A.x, b00, neg(sa), b10), p01 = turn(A.x, b01, neg(sa), b11);
              const float2 p10 = turn(A.x, b10, conj(sa), b00), p11 = turn(A.x, b11, conj(sa), b01);
              // columns: x' = c x - conj(s) y, y' = s x + c y
              auto put = [&](int row, int col, const float2& v) {
                Gb[row * GLD + col] = v;
                Gb[col * GLD + row] = conj(v);
              };
              put(i, k2, turn(B.x, p00, neg(conj(sb)), p01));
              put(i, l2, turn(B.x, p01, sb, p00));
              put(j, k2, turn(B.x, p10, neg(conj(sb)), p11));
              put(j, l2, turn(B.x, p11, sb, p10));
            }
          } else if (warp == 4) {
            if (r + 1 < PM) {
              // entry (m, n) of the next round's pair: row and column of it are
              // each turned with their partner m ^ r, n ^ r of this round
              const Ahead at = ahead;
              const float4 A = rot[at.pm], B = rot[at.pn];
              const float2 g0 = Ga[at.mn], g1 = Ga[at.mn_], g2 = Ga[at.m_n], g3 = Ga[at.m_n_];
              const float am = Ga[at.mm].x, an = Ga[at.nn].x;
              ahead = Ahead(r + 1, tx);             // in the shadow of the chain below
              // the same operations as the update's, so that both see one G
              const float2 fa = make_float2(at.sm * A.y, -A.z), fb = make_float2(at.sn * B.y, B.z);
              float2 g = turn(B.x, turn(A.x, g0, fa, g2), fb, turn(A.x, g1, fa, g3));
              float al = fmaf(at.sm, A.w, am), be = fmaf(at.sn, B.w, an);
              if (at.swap) {
                const float t = al;
                al = be;
                be = t;
                g.y = -g.y;
              }
              float4 q;
              q.w = rotation(al, be, g, q.x, q.y, q.z, off);
              if (lane < PB) s_rot[(r + 1) & 1][tx] = q;
            }
          } else {
            const float4 A = rot[tx];
            const int m = first(tx), n = m ^ r;
            if (warp == 5) {
              if (lane < PB) {
                const float2 g = Ga[m * GLD + n];
                const float al = Ga[m * GLD + m].x, be = Ga[n * GLD + n].x;
                const float2 z = A.y != 0.f || A.z != 0.f ? make_float2(0.f, 0.f) : g;
                Gb[m * GLD + m] = make_float2(al - A.w, 0.f);
                Gb[n * GLD + n] = make_float2(be + A.w, 0.f);
                Gb[m * GLD + n] = z;
                Gb[n * GLD + m] = make_float2(z.x, -z.y);
              }
            } else {
              turn_q<4, 4>(QT + (2 * (warp - 6) + (lane >> 4)) * QLD, m, n, A);
            }
          }
          __syncthreads();
          float2* const t = Ga;
          Ga = Gb;
          Gb = t;
        }
        if (warp == 4 && lane < PB) atomicMax(&s_off, __float_as_int(off));
        // ---- heavier rows first
        if (tid < PM) {
          const float di = Ga[tid * GLD + tid].x;
          int pos = 0;
          for (int j = 0; j < PM; ++j) {
            const float dj = Ga[j * GLD + j].x;
            pos += (dj > di) || (dj == di && j < tid);
          }
          s_pos[tid] = pos;
        }
        __syncthreads();
        if (tid == 0 && rank == 0) atomicMax(st + C_OFF + sw, (unsigned int)s_off);
        // ---- rows <- Q rows: warp w the rows 8 (w % 4).., 32 columns at a time
        const int r0 = 8 * (warp & 3);
        for (int c0 = 0; c0 < lc; c0 += a.chunk) {
          const int n = min(a.chunk, lc - c0);
          if (!resident) {
            __syncthreads();
            stage(u, v, c0, n);
            __syncthreads();
          }
          // a lane takes 1 to 4 columns 64 apart, so that the reads of Q are
          // shared by as many products as the chunk has
          for (int cb = 0; cb < n; cb += 256) {
            const int left = n - cb;
            if (left > 192) apply_rows<4>(a, S, QT, s_pos, ld, cb, n, r0, u, v, rank, c0);
            else if (left > 128) apply_rows<3>(a, S, QT, s_pos, ld, cb, n, r0, u, v, rank, c0);
            else if (left > 64) apply_rows<2>(a, S, QT, s_pos, ld, cb, n, r0, u, v, rank, c0);
            else apply_rows<1>(a, S, QT, s_pos, ld, cb, n, r0, u, v, rank, c0);
          }
        }
        __syncthreads();
        if (tid == 0) {
          publish_block(a.ver + u * 8 + rank, step + 1);
          publish_block(a.ver + v * 8 + rank, step + 1);
        }
      }
    }
    // ---- every block has been through the sweep
    cl.sync();
    passed += (unsigned int)ncl;
    if (rank == 0 && tid == 0) s_ok = leader_barrier(st, passed) ? 1 : 0;
    cl.sync();
    if (*cl.map_shared_rank(&s_ok, 0) == 0) break;
    if (blockIdx.x == 0 && tid == 0) st[C_SWEEPS] = (unsigned int)(sw + 1);
    if (__int_as_float((int)__ldcg(st + C_OFF + sw)) <= kStop32) break;
  }
  cl.sync();                    // s_ok of the first CTA stays readable until here
}

constexpr int RT = 128;                       // threads of the row kernels

// Row i of R32 = R / |R|_F with zero padding, of V = I, and rexp[i] with
// 2^rexp[i] above the largest entry of row i of R, at most twice it.
__global__ void __launch_bounds__(RT)
k_pre_init(const cplx* __restrict__ R, int p, const double* anorm2, Pre32 a, int* rexp) {
  const double n2 = *anorm2;
  const double s = n2 > 0.0 && isfinite(n2) ? rsqrt(n2) : 0.0;
  const int i = blockIdx.x;
  unsigned long long mx = 0ull;
  for (int c = threadIdx.x; c < a.pl; c += RT) {
    float2 v = make_float2(0.f, 0.f);
    if (i < a.k && c < p) {
      const cplx x = R[(long long)i * p + c];
      v = make_float2((float)(x.x * s), (float)(x.y * s));
      mx = max(mx, (unsigned long long)__double_as_longlong(fmax(fabs(x.x), fabs(x.y))));
    }
    a.R[(long long)i * a.pl + c] = v;
  }
  for (int c = threadIdx.x; c < a.vl; c += RT)
    a.V[(long long)i * a.vl + c] = make_float2(i == c ? 1.f : 0.f, 0.f);
  if (i >= a.k) return;
  // the exponent field of the largest magnitude orders like it
  const int e = __reduce_max_sync(0xffffffffu, (int)(mx >> 52));
  __shared__ int sh[RT / 32];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    int m = 0;
#pragma unroll
    for (int w = 0; w < RT / 32; ++w) m = max(m, sh[w]);
    rexp[i] = m == 0 ? 0 : m - 1022;
  }
}

__global__ void k_pre_export(Pre32 a, cplx* __restrict__ V) {
  const long long tot = (long long)a.k * a.k;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
       e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e / a.k), c = (int)(e - (long long)i * a.k);
    const float2 v = a.V[(long long)i * a.vl + c];
    V[e] = cmake(v.x, v.y);
  }
}

__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[RT / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
#pragma unroll
  for (int w = 0; w < RT / 32; ++w) s += sh[w];
  return s;
}

// The largest row sum over the blocks, in *word; the last block to finish
// gets true (and sees every contribution).  Row sums are not negative, so
// their bit patterns order like them, and a NaN is above them all.
__device__ __forceinline__ bool max_over_blocks(double v, unsigned int* ctl, int word) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    atomicMax(reinterpret_cast<unsigned long long*>(ctl + word),
              (unsigned long long)__double_as_longlong(v));
    __threadfence();
    last = atomicAdd(ctl + C_COUNT, 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  return last;
}

constexpr double kDeltaMax = 1e-2;            // |V V^H - I|_inf of a usable V
constexpr double kDeltaEnd = 1e-8;            // below this one more step is the last

// M = V V^H becomes the Newton-Schulz correction -(M - I) / 2, which leaves
// 3/4 |M - I|^2.  The first step decides whether V is usable (then three steps
// reach rounding), the second whether a third is needed.
__global__ void __launch_bounds__(RT) k_pre_orth(cplx* M, int k, unsigned int* ctl, int step) {
  if (step > 0 && ctl[step == 1 ? C_OK : C_GN] == 0u) return;
  const int i = blockIdx.x;
  double s = 0.0;
  for (int j = threadIdx.x; j < k; j += RT) {
    cplx v = M[(long long)i * k + j];
    if (j == i) v.x -= 1.0;
    s += fabs(v.x) + fabs(v.y);
    M[(long long)i * k + j] = cmake(-0.5 * v.x, -0.5 * v.y);
  }
  s = block_sum(s);
  if (step > 1) return;
  if (max_over_blocks(s, ctl, C_DELTA) && threadIdx.x == 0) {
    unsigned long long* w = reinterpret_cast<unsigned long long*>(ctl + C_DELTA);
    const double d = __longlong_as_double((long long)__ldcg(w));
    if (step == 0) ctl[C_OK] = d < kDeltaMax && ctl[C_ERR] == 0u ? 1u : 0u;
    else ctl[C_GN] = d > kDeltaEnd ? 1u : 0u;
    ctl[C_COUNT] = 0u;
    *w = 0ull;
  }
}

__global__ void k_copy_if(cplx* y, const cplx* x, long long n, const unsigned int* flag, int want) {
  if ((*flag != 0u) != (want != 0)) return;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x)
    y[e] = x[e];
}

constexpr double kPairTan = 2.5e-4;           // tangents above this are left to the Jacobi

// E from G = S S^H: E_ij = -sign(D) t g_ij / |g_ij| (D = G_jj - G_ii, t the tangent of
// the rotation that makes the pair orthogonal), exactly anti-Hermitian because
// both halves come from the upper triangle; rexp[i] with 2^rexp[i] next to |S_i|.
// The last block sets the gates of what follows from nu = |E|_inf: E^2 counts above
// 4e-9, E^4 above 1e-4.
__global__ void __launch_bounds__(RT)
k_pre_corr(const cplx* __restrict__ G, int k, double tol, const double* anorm2, double skip_rel,
           double nu_max, cplx* __restrict__ E, int* rexp, unsigned int* ctl) {
  const int i = blockIdx.x;
  const double skip = skip_rel * *anorm2;
  const double al = G[(long long)i * k + i].x;
  if (threadIdx.x == 0)
    rexp[i] = al > 0.0 ? (((int)((unsigned long long)__double_as_longlong(al) >> 52) - 1023) >> 1) + 1 : 0;
  double s = 0.0;
  for (int j = threadIdx.x; j < k; j += RT) {
    cplx e = cmake(0.0, 0.0);
    if (j != i) {
      const double be = G[(long long)j * k + j].x;
      const cplx g = i < j ? G[(long long)i * k + j] : cconj(G[(long long)j * k + i]);
      const double g2 = fma(g.x, g.x, g.y * g.y);
      if (g2 > tol * tol * al * be && g2 > 0.0 && (al > skip || be > skip)) {
        // (i < j) D and sign as the upper element has them
        const double D = i < j ? be - al : al - be;
        const double u = 2.0 / (fabs(D) + sqrt(fma(D, D, 4.0 * g2)));
        if (u * u * g2 < kPairTan * kPairTan) {
          const double c = (D >= 0.0) == (i < j) ? -u : u;
          e = cmake(c * g.x, c * g.y);
          s += u * sqrt(g2);
        }
      }
    }
    E[(long long)i * k + j] = e;
  }
  s = block_sum(s);
  if (max_over_blocks(s, ctl, C_NU) && threadIdx.x == 0) {
    unsigned long long* w = reinterpret_cast<unsigned long long*>(ctl + C_NU);
    const double nu = __longlong_as_double((long long)__ldcg(w));
    const bool on = nu > 0.0 && nu <= nu_max;
    ctl[C_GE] = on;
    ctl[C_GW] = on && nu > 4e-9;
    ctl[C_GW2] = on && nu > 1e-4;
    ctl[C_COUNT] = 0u;
    *w = 0ull;
  }
}

// E <- E + W / 2 - W2 / 8 (W = E^2, W2 = E^4)
__global__ void k_pre_comb(cplx* E, const cplx* W, const cplx* W2, long long n,
                           const unsigned int* ctl) {
  const bool w = ctl[C_GW] != 0u, w2 = ctl[C_GW2] != 0u;
  if (!w) return;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    cplx v = cadd(E[e], cscale(W[e], 0.5));
    if (w2) v = cadd(v, cscale(W2[e], -0.125));
    E[e] = v;
  }
}

// flag[i] = 1 if row i belongs to a pair that is not orthogonal to tol.  For a
// pair of which one row is below the skip weight (it can never be kept), what
// counts is what its rotation would change in the heavier row, as in the
// Jacobi's own stopping rule.  All rows if V was dropped.
__global__ void __launch_bounds__(RT)
k_pre_flag(const cplx* __restrict__ G, int k, double tol, const double* anorm2, double skip_rel,
           int* flag, const unsigned int* ctl) {
  const int i = blockIdx.x;
  const double skip = skip_rel * *anorm2;
  const double al = G[(long long)i * k + i].x;
  int need = ctl[C_OK] == 0u;
  for (int j = threadIdx.x; j < k; j += RT) {
    if (j == i) continue;
    const double be = G[(long long)j * k + j].x;
    const cplx g = i < j ? G[(long long)i * k + j] : G[(long long)j * k + i];
    const double g2 = fma(g.x, g.x, g.y * g.y);
    if (al > skip && be > skip) {
      if (g2 > tol * tol * al * be) need = 1;
    } else if (al > skip || be > skip) {
      const double D = be - al, lo = fmin(al, be), hi = fmax(al, be);
      const double u = 2.0 / (fabs(D) + sqrt(fma(D, D, 4.0 * g2)));
      if (g2 > 0.0 && u * u * g2 * lo > tol * tol * hi) need = 1;
    }
  }
  need = __syncthreads_or(need);
  if (threadIdx.x == 0) flag[i] = need;
}

// act[0] = number of flagged rows, act[1..] their indices in order (one block)
__global__ void __launch_bounds__(1024) k_pre_compact(const int* flag, int k, int* act) {
  __shared__ int wsum[32];
  __shared__ int base;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) base = 0;
  __syncthreads();
  for (int i0 = 0; i0 < k; i0 += 1024) {
    const int i = i0 + threadIdx.x;
    const bool f = i < k && flag[i] != 0;
    const unsigned int m = __ballot_sync(0xffffffffu, f);
    if (lane == 0) wsum[w] = __popc(m);
    __syncthreads();
    int before = base;
    for (int x = 0; x < w; ++x) before += wsum[x];
    if (f) act[1 + before + __popc(m & ((1u << lane) - 1u))] = i;
    __syncthreads();
    if (threadIdx.x == 0)
      for (int x = 0; x < 32; ++x) base += wsum[x];
    __syncthreads();
  }
  if (threadIdx.x == 0) act[0] = base;
}

int grid_for(long long tot) {
  long long g = (tot + 255) / 256;
  return (int)(g > 1216 ? 1216 : g < 1 ? 1 : g);
}

long long round_up(long long x, long long m) { return (x + m - 1) / m * m; }

// Padded rows, and row strides that leave room for the last CTA's share of
// columns (a multiple of 4 per CTA, up to 8 CTAs).
struct PreDims {
  int kp, pl, vl;
};
PreDims pre_dims(int k, int p) {
  const int kp = (int)round_up(k, PM);
  return {kp, (int)round_up(p, 4) + 32, kp + 32};
}
// control words, then the blocks' step counts
size_t ctl_bytes(const PreDims& d) { return (size_t)(C_WORDS + d.kp / PB * 8) * sizeof(int); }
int share(int columns, int C) { return 4 * ((columns + 4 * C - 1) / (4 * C)); }

constexpr size_t kFixedSmem = (size_t)PM * (4 * GLD + QLD) * sizeof(float2);
constexpr int kChunkMax = 640;                // columns staged at once: 32 x 642 x 8 B = 164 KB
constexpr size_t kOwnSmSmem = 116 * 1024;     // more than half of an SM's shared memory

// Clusters of C CTAs that can be resident at once, per device and C (0: not asked yet;
// two host threads may ask at once and get the same answer).  Asked at the largest
// shared memory: every size in use is more than half of an SM's, so the answer is one
// CTA per SM for all of them.
constexpr size_t kMaxSmem = kFixedSmem + (size_t)PM * (kChunkMax + 2) * sizeof(float2);
constexpr int kMaxCluster = 8, kMaxDevices = 64;
std::atomic<int> g_capacity[kMaxDevices][kMaxCluster + 1];
std::atomic<long long> g_queries{0};

void launch_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, int grid, int C, size_t smem,
                   cudaStream_t st, bool coop) {
  *cfg = cudaLaunchConfig_t();
  cfg->gridDim = dim3(grid);
  cfg->blockDim = dim3(PT);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeCooperative;
  at[1].val.cooperative = 1;
  cfg->attrs = at;
  cfg->numAttrs = coop ? 2 : 1;
}

cudaError_t cluster_capacity(int C, int* n) {
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  std::atomic<int>& known = g_capacity[dev % kMaxDevices][C];
  *n = known.load();
  if (*n > 0) return cudaSuccess;
  err = cudaFuncSetAttribute(k_jacobi32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[2];
  launch_config(&cfg, at, C * 1024, C, kMaxSmem, nullptr, false);
  g_queries.fetch_add(1);
  err = cudaOccupancyMaxActiveClusters(n, k_jacobi32, &cfg);
  if (err != cudaSuccess) return err;
  known.store(*n);
  return cudaSuccess;
}

}  // namespace

cudaError_t svd_pre_rotations(int n, const float* al, const float* be, const float* g, float* c,
                              float* s, cudaStream_t st) {
  if (n < 1) return cudaSuccess;
  count_launches(1);
  k_rotations<<<grid_for(n), 256, 0, st>>>(n, al, be, reinterpret_cast<const float2*>(g), c,
                                           reinterpret_cast<float2*>(s));
  return cudaGetLastError();
}

long long svd_pre_queries() { return g_queries.load(); }

size_t svd_pre_bytes(int k, int p) {
  const PreDims d = pre_dims(k, p);
  return (size_t)d.kp * (d.pl + d.vl) * sizeof(float2) + 4 * (size_t)k * k * sizeof(cplx) +
         (size_t)(3 * k + 1) * sizeof(int) + ctl_bytes(d) + 6 * 256;
}

SvdPre svd_pre_carve(void* ws, int k, int p) {
  const PreDims d = pre_dims(k, p);
  char* c = static_cast<char*>(ws);
  SvdPre s;
  auto take = [&](size_t bytes) {
    char* r = c;
    c += round_up((long long)bytes, 256);
    return r;
  };
  s.rows32 = take((size_t)d.kp * (d.pl + d.vl) * sizeof(float2));
  for (cplx*& m : s.K) m = reinterpret_cast<cplx*>(take((size_t)k * k * sizeof(cplx)));
  s.act = reinterpret_cast<int*>(take((size_t)(3 * k + 1) * sizeof(int)));
  s.rexp = s.act + 2 * k + 1;
  s.ctl = reinterpret_cast<unsigned int*>(take(ctl_bytes(d)));
  s.ok = reinterpret_cast<int*>(s.ctl + C_OK);
  s.sweeps = reinterpret_cast<const int*>(s.ctl + C_SWEEPS);
  s.gate_n = reinterpret_cast<int*>(s.ctl + C_GN);
  s.gate = reinterpret_cast<int*>(s.ctl + C_GE);
  s.gate_w = reinterpret_cast<int*>(s.ctl + C_GW);
  s.gate_w2 = reinterpret_cast<int*>(s.ctl + C_GW2);
  return s;
}

cudaError_t svd_pre_rotate(const SvdPre& s, const cplx* R, int k, int p, const double* anorm2,
                           bool expired, cudaStream_t st) {
  const PreDims d = pre_dims(k, p);
  cudaError_t err = cudaMemsetAsync(s.ctl, 0, ctl_bytes(d), st);
  if (err != cudaSuccess) return err;
  if (expired) {
    err = cudaMemsetAsync(s.ctl + C_ERR, 1, sizeof(unsigned int), st);
    if (err != cudaSuccess) return err;
  }
  Pre32 a;
  a.R = static_cast<float2*>(s.rows32);
  a.V = a.R + (size_t)d.kp * d.pl;
  a.k = k;
  a.kp = d.kp;
  a.pl = d.pl;
  a.vl = d.vl;
  a.nb = d.kp / PB;
  a.ver = s.ctl + C_WORDS;
  count_launches(1);
  k_pre_init<<<d.kp, RT, 0, st>>>(R, p, anorm2, a, s.rexp);
  // as many CTAs per pair as give every CTA an SM of its own (two on one SM
  // take turns at every phase of the step)
  const int pairs = a.nb / 2;
  int C = kMaxCluster, cap = 0;
  size_t smem = 0;
  for (;; --C) {
    a.pc = share(p, C);
    a.vc = share(d.kp, C);
    a.chunk = a.pc + a.vc < kChunkMax ? a.pc + a.vc : kChunkMax;
    smem = kFixedSmem + (size_t)PM * (a.chunk + 2) * sizeof(float2);
    if (smem < kOwnSmSmem) smem = kOwnSmSmem;
    err = cluster_capacity(C, &cap);
    if (err != cudaSuccess) return err;
    if (cap >= pairs || C == 1) break;
  }
  if (cap < 1) return cudaErrorInvalidConfiguration;
  const int ncl = pairs < cap ? pairs : cap;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[2];
  launch_config(&cfg, at, ncl * C, C, smem, st, true);
  count_launches(1);
  err = cudaLaunchKernelEx(&cfg, k_jacobi32, a, s.ctl);
  if (err != cudaSuccess) return err;
  count_launches(1);
  k_pre_export<<<grid_for((long long)k * k), 256, 0, st>>>(a, s.K[0]);
  return cudaGetLastError();
}

cudaError_t svd_pre_orth(const SvdPre& s, cplx* M, int k, int step, cudaStream_t st) {
  count_launches(1);
  k_pre_orth<<<k, RT, 0, st>>>(M, k, s.ctl, step);
  return cudaGetLastError();
}

cudaError_t vec_copy_if(cplx* y, const cplx* x, long long n, const int* flag, bool want,
                        cudaStream_t st) {
  count_launches(1);
  k_copy_if<<<grid_for(n), 256, 0, st>>>(y, x, n, reinterpret_cast<const unsigned int*>(flag),
                                         want ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t svd_pre_corr(const SvdPre& s, const cplx* G, int k, double tol, const double* anorm2,
                         double skip_rel, double nu_max, cplx* E, cudaStream_t st) {
  count_launches(1);
  k_pre_corr<<<k, RT, 0, st>>>(G, k, tol, anorm2, skip_rel, nu_max, E, s.rexp, s.ctl);
  return cudaGetLastError();
}

cudaError_t svd_pre_comb(const SvdPre& s, cplx* E, const cplx* W, const cplx* W2, int k,
                         cudaStream_t st) {
  const long long n = (long long)k * k;
  count_launches(1);
  k_pre_comb<<<grid_for(n), 256, 0, st>>>(E, W, W2, n, s.ctl);
  return cudaGetLastError();
}

cudaError_t svd_pre_list(const SvdPre& s, const cplx* G, int k, double tol, const double* anorm2,
                         double skip_rel, cudaStream_t st) {
  int* flag = s.act + k + 1;
  count_launches(2);
  k_pre_flag<<<k, RT, 0, st>>>(G, k, tol, anorm2, skip_rel, flag, s.ctl);
  k_pre_compact<<<1, 1024, 0, st>>>(flag, k, s.act);
  return cudaGetLastError();
}

}  // namespace ite
