// Batched complex FP64 GEMM with arbitrary element strides, used by every
// tensor contraction of the FP64 path (two-site H_eff, environments, local
// right-hand sides, two-site merges).
//
// On GB300 the FP64 pipe issues about two DFMA per clock per SM (measured
// 1.19 TFLOP/s for the whole GPU), so these kernels are bound by that pipe, and
// what a shape costs is the work of its busiest SM: shared-memory and L2 traffic
// are far below their limits even for 8 x 8 tiles.  Three tile sizes, all of 256
// threads:
//   32 x 32, 2 x 2 outputs per thread, where the tiles are many;
//   16 x 16, one output per thread;
//   8 x 8, K dealt to four groups of 64 threads whose sums are added in order.
// Small products (chi = 64: 256 x 64 x 320) made 16 tiles of 32 x 32, 136 of 152
// SMs idle: 347 us, against 33 us of FP64 work spread over the GPU.  One small
// H_eff (chi = 32) 250 -> 55 us, GMRES(10) at chi = 64 5.55 -> 1.91 ms (with the
// MPO mix's change).
#include <atomic>

#include "common.cuh"

namespace ite {
namespace {

constexpr int BM = 32, BN = 32, BK = 8, THREADS = 256;

template <bool CONJ_A, bool CONJ_B>
__global__ void __launch_bounds__(THREADS)
zgemm_kernel(GemmArgs g, bool a_kfast, bool b_nfast) {
  __shared__ cplx As[BK][BM + 1];
  __shared__ cplx Bs[BK][BN + 1];
  if (g.run_if && *g.run_if == 0) return;
  const int t = threadIdx.x;
  const int tx = t % 16, ty = t / 16;
  const int row0 = blockIdx.y * BM, col0 = blockIdx.x * BN;
  const int b = blockIdx.z;
  const cplx* A = g.A + (long long)b * g.sAb;
  const cplx* B = g.B + (long long)b * g.sBb;

  // load mapping: A tile is BM x BK (256 elements), B tile is BK x BN
  const int ai = a_kfast ? t / BK : t % BM;
  const int ak = a_kfast ? t % BK : t / BM;
  const int bk = b_nfast ? t / BN : t % BK;
  const int bj = b_nfast ? t % BN : t / BK;

  cplx acc[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[i][j] = cmake(0.0, 0.0);

  for (int k0 = 0; k0 < g.K; k0 += BK) {
    {
      const int gi = row0 + ai, gk = k0 + ak;
      cplx v = cmake(0.0, 0.0);
      if (gi < g.M && gk < g.K) {
        v = A[(long long)gi * g.sAm + (long long)gk * g.sAk];
        if (CONJ_A) v = cconj(v);
      }
      As[ak][ai] = v;
    }
    {
      const int gk = k0 + bk, gj = col0 + bj;
      cplx v = cmake(0.0, 0.0);
      if (gk < g.K && gj < g.N) {
        v = B[(long long)gk * g.sBk + (long long)gj * g.sBn];
        if (CONJ_B) v = cconj(v);
      }
      Bs[bk][bj] = v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      const cplx a0 = As[k][ty * 2], a1 = As[k][ty * 2 + 1];
      const cplx b0 = Bs[k][tx * 2], b1 = Bs[k][tx * 2 + 1];
      cfma(acc[0][0], a0, b0);
      cfma(acc[0][1], a0, b1);
      cfma(acc[1][0], a1, b0);
      cfma(acc[1][1], a1, b1);
    }
    __syncthreads();
  }

  cplx* C = g.C + (long long)b * g.sCb;
  const cplx* Z = g.Z ? g.Z + (long long)b * g.sCb : nullptr;
  const bool use_beta = (g.beta.x != 0.0 || g.beta.y != 0.0);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int r = row0 + ty * 2 + i;
    if (r >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = col0 + tx * 2 + j;
      if (c >= g.N) continue;
      const long long idx = (long long)r * g.ldc + c;
      cplx v = cmul(g.alpha, acc[i][j]);
      if (use_beta) v = cadd(v, cmul(g.beta, C[idx]));
      if (Z) v = cadd(v, cmul(g.gamma, Z[idx]));
      C[idx] = v;
    }
  }
}

// T x T outputs, K dealt to KG groups of T * T threads, 32 terms at a time; the
// next terms are fetched into registers while these are used.
template <int T, int KG, bool CONJ_A, bool CONJ_B>
__global__ void __launch_bounds__(THREADS)
zgemm_small(GemmArgs g, bool a_kfast, bool b_nfast) {
  static_assert(T * T * KG == THREADS, "one output per thread and group");
  constexpr int KC = 32, NL = T * KC / THREADS;       // terms per chunk, loads per thread
  __shared__ cplx As[KC][T + 1];
  __shared__ cplx Bs[KC][T + 1];
  __shared__ cplx red[KG > 1 ? (KG - 1) * T * T : 1];
  if (g.run_if && *g.run_if == 0) return;
  const int t = threadIdx.x;
  const int row0 = blockIdx.y * T, col0 = blockIdx.x * T, b = blockIdx.z;
  const cplx* A = g.A + (long long)b * g.sAb;
  const cplx* B = g.B + (long long)b * g.sBb;
  const int o = t % (T * T), kg = t / (T * T), oi = o / T, oj = o % T;
  cplx ra[NL], rb[NL];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      const int e = t + l * THREADS;
      const int ai = a_kfast ? e / KC : e % T, ak = a_kfast ? e % KC : e / T;
      const int bj = b_nfast ? e % T : e / KC, bk = b_nfast ? e / T : e % KC;
      ra[l] = rb[l] = cmake(0.0, 0.0);
      if (row0 + ai < g.M && k0 + ak < g.K)
        ra[l] = A[(long long)(row0 + ai) * g.sAm + (long long)(k0 + ak) * g.sAk];
      if (col0 + bj < g.N && k0 + bk < g.K)
        rb[l] = B[(long long)(k0 + bk) * g.sBk + (long long)(col0 + bj) * g.sBn];
    }
  };
  cplx acc = cmake(0.0, 0.0);
  fetch(0);
  for (int k0 = 0; k0 < g.K; k0 += KC) {
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      const int e = t + l * THREADS;
      const int ai = a_kfast ? e / KC : e % T, ak = a_kfast ? e % KC : e / T;
      const int bj = b_nfast ? e % T : e / KC, bk = b_nfast ? e / T : e % KC;
      As[ak][ai] = CONJ_A ? cconj(ra[l]) : ra[l];
      Bs[bk][bj] = CONJ_B ? cconj(rb[l]) : rb[l];
    }
    __syncthreads();
    if (k0 + KC < g.K) fetch(k0 + KC);
    const int n = min(KC, g.K - k0);
    if (n == KC) {
#pragma unroll
      for (int k = 0; k < KC / KG; ++k) cfma(acc, As[kg + KG * k][oi], Bs[kg + KG * k][oj]);
    } else {
      for (int k = kg; k < n; k += KG) cfma(acc, As[k][oi], Bs[k][oj]);
    }
    __syncthreads();
  }
  if (KG > 1) {
    if (kg > 0) red[(kg - 1) * T * T + o] = acc;
    __syncthreads();
    if (kg > 0) return;
#pragma unroll
    for (int i = 0; i + 1 < KG; ++i) acc = cadd(acc, red[i * T * T + o]);
  }
  const int r = row0 + oi, c = col0 + oj;
  if (r >= g.M || c >= g.N) return;
  const long long idx = (long long)b * g.sCb + (long long)r * g.ldc + c;
  cplx v = cmul(g.alpha, acc);
  if (g.beta.x != 0.0 || g.beta.y != 0.0) v = cadd(v, cmul(g.beta, g.C[idx]));
  if (g.Z) v = cadd(v, cmul(g.gamma, g.Z[idx]));
  g.C[idx] = v;
}

template <int T, bool CA, bool CB>
void launch(const GemmArgs& g, bool a_kfast, bool b_nfast, cudaStream_t st) {
  const dim3 grid((g.N + T - 1) / T, (g.M + T - 1) / T, g.batch);
  if constexpr (T == 32) zgemm_kernel<CA, CB><<<grid, THREADS, 0, st>>>(g, a_kfast, b_nfast);
  else zgemm_small<T, 256 / (T * T), CA, CB><<<grid, THREADS, 0, st>>>(g, a_kfast, b_nfast);
}

template <int T>
void launch_conj(const GemmArgs& g, bool a_kfast, bool b_nfast, cudaStream_t st) {
  if (g.conjA && g.conjB) launch<T, true, true>(g, a_kfast, b_nfast, st);
  else if (g.conjA) launch<T, true, false>(g, a_kfast, b_nfast, st);
  else if (g.conjB) launch<T, false, true>(g, a_kfast, b_nfast, st);
  else launch<T, false, false>(g, a_kfast, b_nfast, st);
}

// Work of the busiest SM in outputs, if the tiles are dealt evenly, with what a
// small tile costs more per output (fewer products per load).
double busiest(const GemmArgs& g, int T, double factor, int sms) {
  const double tiles = (double)((g.M + T - 1) / T) * ((g.N + T - 1) / T) * g.batch;
  return factor * T * T * (double)(long long)((tiles + sms - 1.0) / sms);
}

// C shares memory with A or B (as intervals of addresses).
bool in_place(const GemmArgs& g) {
  struct Span { const cplx *lo, *hi; };
  auto span = [&](const cplx* p, long long n0, long long s0, long long n1, long long s1,
                  long long sb) {
    Span r = {p, p + 1};
    const long long d[3] = {(n0 - 1) * s0, (n1 - 1) * s1, (g.batch - 1) * sb};
    for (long long x : d) (x < 0 ? r.lo : r.hi) += x;
    return r;
  };
  const Span a = span(g.A, g.M, g.sAm, g.K, g.sAk, g.sAb), b = span(g.B, g.K, g.sBk, g.N, g.sBn, g.sBb);
  const Span c = span(g.C, g.M, g.ldc, g.N, 1, g.sCb);
  return (c.lo < a.hi && a.lo < c.hi) || (c.lo < b.hi && b.lo < c.hi);
}

}  // namespace

cudaError_t device_sms(int* sms) {
  static std::atomic<int> known[64];
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  *sms = known[dev & 63].load();
  if (*sms > 0) return cudaSuccess;
  err = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  if (err == cudaSuccess) known[dev & 63].store(*sms);
  return err;
}

cudaError_t zgemm(const GemmArgs& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
  if (g.batch > 65535 || (g.M + BM - 1) / BM > 65535) return cudaErrorInvalidValue;
  const bool a_kfast = (g.sAk == 1);
  const bool b_nfast = (g.sBn == 1) || (g.sBk != 1);
  int sms = 0;
  const cudaError_t err = device_sms(&sms);
  if (err != cudaSuccess) return err;
  const double w32 = busiest(g, 32, 1.0, sms), w16 = busiest(g, 16, 1.1, sms),
               w8 = busiest(g, 8, 1.25, sms);
  // a product of one 32 x 32 tile reads its operands in full before it writes, so it
  // may write over one of them; smaller tiles would read what others have written
  const bool one_tile = g.M <= BM && g.N <= BN && in_place(g);
  count_launches(1);
  if ((w32 <= w16 && w32 <= w8) || (g.M + 7) / 8 > 65535 || one_tile) launch_conj<32>(g, a_kfast, b_nfast, st);
  else if (w16 <= w8) launch_conj<16>(g, a_kfast, b_nfast, st);
  else launch_conj<8>(g, a_kfast, b_nfast, st);
  return cudaGetLastError();
}

}  // namespace ite
