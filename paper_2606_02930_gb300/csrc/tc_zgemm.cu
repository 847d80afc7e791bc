// FP64-accurate complex GEMM on the bf16 tensor cores by exact slicing.
//
// GB300 runs FP64 at about 1.2 TFLOP/s but bf16 MMA at about 2 PFLOP/s, so the
// contractions of the FP64 path are computed as sums of exact bf16 products:
//
//  * complex C = op(A) op(B) becomes the real product of the row-embedded
//    A^ (rows 2r, 2r+1 = [Re, -Im], [Im, Re] interleaved along K) with the
//    K-major B^T (rows = columns of B, (Re, Im) interleaved along K);
//  * every row of A^ and every row of B^T is scaled by its own power of two
//    2^e (largest magnitude < 2^e), rounded to the nearest multiple of
//    2^(e-56) (error <= 2^(e-57)) and cut into S = 8 balanced base-128
//    digits, x = 2^e sum_p a_p 2^(-7p) with a_1 in [-128, 128] and the lower
//    digits in [-64, 64], zero-centred so that the rounding and the dropped
//    products below are unbiased.  Each digit is exact in bf16.  The slicing
//    uses integer operations on the bit patterns only;
//  * digit products a_p b_q of the same weight d = p + q are accumulated by
//    tcgen05.mma in one fp32 TMEM accumulator per d = 2..S+1 over K-chunks of
//    256 real terms: |a_1 b_1| <= 2^14 and every other product is at most
//    2^13, so every partial sum is an integer of magnitude below
//    256 (2 2^13 + (S-2) 2^12) < 2^24 and fp32 accumulation is exact;
//  * after each chunk the epilogue warps convert the accumulators to integers
//    and add them exactly into two int64 registers per output
//    (hi = sum_{d<=4} v_d 2^(7(4-d)), lo = sum_{d>=5} v_d 2^(7(S+1-d))); the
//    result is 2^(eA+eB) (hi 2^-28 + lo 2^-7(S+1)), rounded once to FP64.
//  Products of weight d > S+1 are dropped (both digits are low ones: at most
//  (S-1) 2^12 2^(-7(S+2)) < 2^-55 per term, of either sign); with the
//  rounding this gives an error below about K 2^-54 |A_row| |B_col|
//  (max-norms) in the worst case and about sqrt(K) of that for unrelated
//  terms: FP64-class, at the rounding level of an FP64 product of the same
//  length.
//
// Tiles: 128 real rows x BN columns, K tiles of 32 (64-byte swizzle); a ring
// of 2 stages each holding the 8 digit tiles of A and of B.  The accumulators
// of the 8 weights lie side by side in TMEM (8 BN columns), and so do the
// digit tiles of B in shared memory: digit a_p against the stacked digits
// b_1..b_{S+1-p} is one MMA of N = (S+1-p) BN that adds to the weights
// p+1..S+1, so a K step of 16 takes 8 (BN = 32) wide MMAs instead of 36 of
// N = 32, which ran at 109 clocks each (3.8 us per K tile, 0.56 us of it MMA
// work) because a narrow MMA still reads all of its A tile.
//   BN = 32: two sets of accumulators (512 columns), the epilogue of one chunk
//            overlaps the MMAs of the next; 80 KB per K tile and 128 x 32;
//   BN = 64: one set; 96 KB per K tile and 128 x 64, less shared-memory fill
//            per product, for products with enough tiles for every SM.
// Persistent over the tiles of all batch entries.  Epilogue warps (two TMEM
// lane quarters' worth per 32 columns), one TMA producer warp, one MMA warp.
// All waits are bounded.
#include <cuda_bf16.h>

#include <cstdint>

#include <atomic>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace ite {
namespace {

using namespace tc;

constexpr int S = 8;
constexpr int BM = 128, BK = 32;
constexpr int KC = 256;                         // real K terms per exact chunk
constexpr int KB_PER_CHUNK = KC / BK;
constexpr int STAGES = 2;
static_assert(S == 8, "the epilogue's lo word is scaled by 2^-7(S+1) = 2^-63");
static_assert(KC * (2 * (1 << 13) + (S - 2) * (1 << 12)) < (1 << 24) && KC * (1 << 14) < (1 << 24),
              "chunk sums must stay exact in fp32");
constexpr uint32_t A_SLICE = BM * BK * 2;       // 8 KB

template <int BN>
struct Tile {
  static constexpr int BUFS = BN == 32 ? 2 : 1;           // accumulator sets
  static constexpr int ACC = S * BN;                      // columns of one set
  static constexpr int EW = 4 * (BN / 32);                // epilogue warps
  static constexpr int THREADS = 32 * (EW + 2);
  static constexpr uint32_t B_SLICE = BN * BK * 2;
  static constexpr uint32_t STAGE = S * (A_SLICE + B_SLICE);
  static constexpr size_t SMEM = 1024 + STAGES * STAGE + (2 * STAGES + 4) * 8 + 16;
  static_assert(BUFS * ACC == 512, "all of TMEM");
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// box of all digits: (k, row, batch entry, digit)
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, uint64_t* bar, int x,
                                            int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::
          "r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(0), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ double pow2(int e) {
  // 2^e for -1022 <= e <= 1023 built from the bit pattern
  if (e < -1022) return 0.0;
  if (e > 1023) e = 1023;
  return __longlong_as_double((long long)(e + 1023) << 52);
}

// (hi 2^-28 + lo 2^-63) 2^e rounded once to nearest even, in integer
// arithmetic: the FP64 pipe issues two lanes per clock and SM, so the
// conversions and products of the floating-point form took longer than the
// MMAs of a short K.
__device__ __forceinline__ double scaled_sum(long long hi, long long lo, int e) {
  // T = hi 2^35 + lo, 128 bits
  unsigned long long l = (unsigned long long)hi << 35;
  long long h = hi >> 29;
  l += (unsigned long long)lo;
  h += (lo >> 63) + (l < (unsigned long long)lo ? 1 : 0);
  const bool neg = h < 0;
  unsigned long long uh = (unsigned long long)h;
  if (neg) {
    l = ~l + 1ull;
    uh = ~uh + (l == 0ull ? 1ull : 0ull);
  }
  if ((uh | l) == 0ull) return 0.0;
  int top = 127;                               // index of the leading bit
  if (uh == 0ull) {
    uh = l;
    l = 0ull;
    top = 63;
  }
  const int z = __clzll((long long)uh);
  top -= z;
  if (z) {
    uh = (uh << z) | (l >> (64 - z));
    l <<= z;
  }
  unsigned long long m = uh >> 11;
  const unsigned int rem = (unsigned int)uh & 0x7FFu;
  m += (rem > 0x400u || (rem == 0x400u && (l != 0ull || (m & 1ull)))) ? 1ull : 0ull;
  const int E = top - 63 + e + 1023;           // biased exponent of the leading bit
  double r;
  if (E >= 1 && E <= 2045) {
    r = __longlong_as_double((long long)(((unsigned long long)(E - 1) << 52) + m));
  } else {
    r = (double)m * pow2(top - 63 - 52) * pow2(e);       // at the ends of the range
  }
  return neg ? -r : r;
}

struct EmuShape {
  int Mr, N, nkb;                              // real rows, columns, K tiles
  int mt, nt, tiles;                           // tiles per batch entry, and in all
  int a_batched, b_batched;
  long long ldc, sCb;
  cplx alpha, beta, gamma;
  cplx* C;
  const cplx* Z;
  const int *eA, *eB;
  const int* run_if;
  int* err;
};

template <int BN>
__global__ void __launch_bounds__(Tile<BN>::THREADS, 1)
k_zgemm_slices(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ EmuShape g) {
  typedef Tile<BN> T;
  if (g.run_if && *g.run_if == 0) return;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * T::STAGE);
  uint64_t* empty = full + STAGES;
  uint64_t* acc_full = empty + STAGES;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  __shared__ int s_fail, s_loads, s_mmas;       // K tiles whose loads, MMAs were issued

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkb = g.nkb;
  const int nchunk = (nkb + KB_PER_CHUNK - 1) / KB_PER_CHUNK;

  if (threadIdx.x == 0) {
    s_fail = s_loads = s_mmas = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], T::EW);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  // tile t: batch entry, row tile, column tile (columns fastest: CTAs that run
  // together share rows of A in L2)
  auto locate = [&](int t, int& b, int& m0, int& n0) {
    n0 = (t % g.nt) * BN;
    t /= g.nt;
    m0 = (t % g.mt) * BM;
    b = t / g.mt;
  };

  if (warp == T::EW) {
    // ---- TMA producer: K tile kb brings the 8 digit tiles of A and of B
    if (lane == 0) {
      int it = 0;
      for (int t = blockIdx.x; t < g.tiles && !*((volatile int*)&s_fail); t += gridDim.x) {
        int b, m0, n0;
        locate(t, b, m0, n0);
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = it % STAGES;
          if (it >= STAGES && !mbar_wait(&empty[s], ((it / STAGES) + 1) & 1)) {
            s_fail = 1;
            break;
          }
          uint8_t* st = smem + s * T::STAGE;
          mbar_expect_tx(&full[s], T::STAGE);
          tma_load_4d(st, &tmA, &full[s], kb * BK, m0, g.a_batched ? b : 0);
          tma_load_4d(st + S * A_SLICE, &tmB, &full[s], kb * BK, n0, g.b_batched ? b : 0);
        }
      }
      s_loads = it;
    }
  } else if (warp == T::EW + 1) {
    // ---- MMA issuer
    if (lane == 0) {
      int it = 0, ch = 0;
      for (int t = blockIdx.x; t < g.tiles && !*((volatile int*)&s_fail); t += gridDim.x) {
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int kin = kb % KB_PER_CHUNK;
          const int buf = ch % T::BUFS, use = ch / T::BUFS;
          if (kin == 0 && use >= 1) {
            if (!mbar_wait(&acc_empty[buf], (use - 1) & 1)) {
              s_fail = 1;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          const int s = it % STAGES;
          if (!mbar_wait(&full[s], (it / STAGES) & 1)) {
            s_fail = 1;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a0 = smem_u32(smem + s * T::STAGE);
          const uint32_t b0 = a0 + S * A_SLICE;
          const uint32_t acc = tmem + buf * T::ACC;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
#pragma unroll
            for (int p = 1; p <= S; ++p) {
              // digit p of A against digits 1..S+1-p of B: weights p+1..S+1
              const uint64_t da = kmajor_desc<BK>(a0 + (p - 1) * A_SLICE + kk * 32);
              const uint32_t accum = (kin == 0 && p == 1 && kk == 0) ? 0u : 1u;
#pragma unroll
              for (int n0 = 0; n0 < (S + 1 - p) * BN; n0 += 256) {
                const int n = (S + 1 - p) * BN - n0 < 256 ? (S + 1 - p) * BN - n0 : 256;
                mma_bf16(acc + (p - 1) * BN + n0, da, kmajor_desc<BK>(b0 + n0 * (BK * 2) + kk * 32),
                         bf16_idesc(n), accum);
              }
            }
          }
          mma_commit(&empty[s]);
          if (kin == KB_PER_CHUNK - 1 || kb == nkb - 1) {
            mma_commit(&acc_full[buf]);
            ++ch;
          }
        }
      }
      s_mmas = it;
    }
  } else {
    // ---- epilogue warps: TMEM lane quarter warp % 4, columns 32 (warp / 4)..
    const int q = warp & 3, cbase = 32 * (warp >> 2);
    const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + cbase;
    const bool beta = g.beta.x != 0.0 || g.beta.y != 0.0;
    const bool unit = g.alpha.x == 1.0 && g.alpha.y == 0.0;
    int ch = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < g.tiles && ok; t += gridDim.x) {
      int b, m0, n0;
      locate(t, b, m0, n0);
      n0 += cbase;
      long long hi[32], lo[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) { hi[j] = 0; lo[j] = 0; }
      for (int c = 0; c < nchunk; ++c, ++ch) {
        const int buf = ch % T::BUFS, use = ch / T::BUFS;
        ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[buf], use & 1) ? 1 : 0) != 0;
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // exact integer accumulation of the chunk
#pragma unroll 1
        for (int dd = 0; dd < S; ++dd) {
          float v[32];
          tmem_ld32(lane_base + buf * T::ACC + dd * BN, v);
          const int d = dd + 2;
          if (d <= 4) {
            const int mul = 1 << (7 * (4 - d));
#pragma unroll
            for (int j = 0; j < 32; ++j) hi[j] += (long long)__float2int_rn(v[j]) * mul;
          } else {
            const int mul = 1 << (7 * (S + 1 - d));
#pragma unroll
            for (int j = 0; j < 32; ++j) lo[j] += (long long)__float2int_rn(v[j]) * mul;
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[buf]);
      }
      if (!ok) break;
      // real row rr, columns n0..: 2^(eA+eB) (hi 2^-28 + lo 2^-7(S+1)).
      // Lanes 2i / 2i+1 hold Re / Im of complex row rr/2: the even lane
      // writes columns 0..15, the odd lane columns 16..31.
      const int rr = m0 + q * 32 + lane, r = rr >> 1;
      const bool row = rr < g.Mr, odd = lane & 1;
      const int ea = row ? g.eA[(g.a_batched ? b * (g.Mr >> 1) : 0) + r] : 0;
      const int* eb = g.eB + (g.b_batched ? (long long)b * g.N : 0);
      cplx* Cb = g.C + (long long)b * g.sCb + (long long)r * g.ldc;
      const cplx* Zb = g.Z ? g.Z + (long long)b * g.sCb + (long long)r * g.ldc : nullptr;
#pragma unroll
      for (int h = 0; h < 16; ++h) {
        const int na = n0 + h, nb = na + 16;
        const double x = scaled_sum(hi[h], lo[h], ea + (na < g.N ? eb[na] : 0));
        const double y = scaled_sum(hi[h + 16], lo[h + 16], ea + (nb < g.N ? eb[nb] : 0));
        // the even lane needs Im of column h, the odd lane Re of column h+16
        const double recv = __shfl_xor_sync(0xffffffffu, odd ? x : y, 1);
        const int n = odd ? nb : na;
        if (row && n < g.N) {
          cplx out = odd ? cmake(recv, y) : cmake(x, recv);
          if (!unit) out = cmul(g.alpha, out);
          if (beta) out = cadd(out, cmul(g.beta, Cb[n]));
          if (Zb) out = cadd(out, cmul(g.gamma, Zb[n]));
          Cb[n] = out;
        }
      }
    }
    if (!ok && lane == 0) s_fail = 1;
  }
  __syncthreads();
  // after a wait that ran out: the last loads and MMAs of each stage (bounded), so that
  // none is in flight when the block's memory is given back
  if (s_fail && threadIdx.x == 0) {
    atomicExch(g.err, 1);
    for (int it = max(s_loads - STAGES, 0); it < s_loads; ++it)
      mbar_wait(&full[it % STAGES], (it / STAGES) & 1);
    for (int it = max(s_mmas - STAGES, 0); it < s_mmas; ++it)
      mbar_wait(&empty[it % STAGES], (it / STAGES) & 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// ------------------------------------------------------------------ slicing
// Magnitude bits of a double (the pattern of |x| orders like |x|).
__device__ __forceinline__ unsigned long long mag_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// exponent e with max magnitude < 2^e, from the largest magnitude pattern
__device__ __forceinline__ int scale_exponent(unsigned long long mb) {
  if (mb == 0) return 0;
  const int E = (int)(mb >> 52);
  if (E == 0) return -1022;                     // subnormal range
  return E - 1023 + 1;
}

// T = |x| 2^(7S - e) rounded to the nearest integer (ties up), from the bit
// pattern.  With max|x| < 2^e the row maximum has a shift of 3 and is exact;
// T < 2^(7S) for every entry of the row.
__device__ __forceinline__ unsigned long long fixed_digits(double x, int e) {
  const unsigned long long b = mag_bits(x);
  const int E = (int)(b >> 52);
  unsigned long long mant = b & 0x000FFFFFFFFFFFFFull;
  int Ee = E;
  if (E == 0) Ee = 1; else mant |= 0x0010000000000000ull;
  const int shift = Ee - 1075 + 7 * S - e;      // |x| = mant 2^(Ee-1075)
  if (shift >= 0) return shift >= 64 ? 0ull : mant << shift;
  const int r = -shift;
  return r >= 64 ? 0ull : (mant + (1ull << (r - 1))) >> r;
}

// Balanced base-128 digits of T as fp32 patterns (bf16 in the upper half):
// T = sum_p g_p 2^(7(S-p)) with the leading g_1 in [0, 128] and g_p in [-64, 63]
// for p >= 2, all negated for x < 0.  Adding 64 to every lower digit of T
// makes its plain base-128 digits g_p + 64.  The low digits are centred on
// zero, so neither the dropped low-weight products nor the rounding give the
// sums a bias toward zero.
__device__ __forceinline__ void balanced_digits(unsigned long long T, bool neg, unsigned int (&f)[S]) {
  unsigned long long bias = 0;
#pragma unroll
  for (int i = 0; i < S - 1; ++i) bias |= 64ull << (7 * i);
  T += bias;
  const unsigned int sign = neg ? 0x80000000u : 0u;
#pragma unroll
  for (int p = 1; p <= S; ++p) {
    const unsigned int g = (unsigned int)(T >> (7 * (S - p))) & (p == 1 ? 0xFFu : 127u);
    // 2^23 + g as a float, minus 2^23 (+ 64): exact, without the conversion unit
    const float v = __uint_as_float(0x4B000000u | g) - (p == 1 ? 8388608.f : 8388672.f);
    f[p - 1] = __float_as_uint(v) ^ sign;
  }
}

// One operand: `rows` rows (rows of A or columns of B) of K complex entries per
// batch entry, element (r, k) at p[b sb + r sr + k sk].
struct Operand {
  const cplx* p;
  long long sr, sk, sb;
  int conj, rows, nb;
  __nv_bfloat16* out;                           // digits: (digit, batch, real row, K)
  int* e;                                       // exponents: (batch, row)
  const int* kexp;                              // entry k times 2^(ksign kexp[k])
  int ksign;
};

// x 2^d by its exponent field (exact; what leaves the normal range at the lower
// end is 0)
__device__ __forceinline__ double shifted(double x, int d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)(b >> 52) & 0x7FF, to = E + d;
  if (E == 0 || E == 0x7FF) return x;
  if (to < 1) return 0.0;
  return __longlong_as_double((long long)((b & 0x800FFFFFFFFFFFFFull) |
                                          (unsigned long long)min(to, 0x7FE) << 52));
}

// entry k of the row of `o` that starts at x (SCALED: kexp counts; an instance of its
// own, because the test alone cost the H_eff's cuts a fifth of their time)
template <bool SCALED>
__device__ __forceinline__ cplx entry(const Operand& o, const cplx* x, int k) {
  cplx v = x[(long long)k * o.sk];
  if (SCALED) {
    const int d = o.ksign * o.kexp[k];
    v = cmake(shifted(v.x, d), shifted(v.y, d));
  }
  return v;
}

constexpr int CR = 8;                           // rows per block

// Writes the digits of element k of row r (both of it, interleaved): rows of B
// as (Re, Im), rows of A as the real rows (Re, -Im) and (Im, Re).
template <bool EMBED>
__device__ __forceinline__ void write_digits(const Operand& o, long long row, long long digit_stride,
                                             int Kp, int k, cplx v, int e) {
  unsigned int fr[S], fi[S];
  balanced_digits(fixed_digits(v.x, e), v.x < 0.0, fr);
  balanced_digits(fixed_digits(v.y, e), (v.y < 0.0) != (o.conj != 0), fi);
  unsigned int* d = reinterpret_cast<unsigned int*>(o.out) + (row * Kp >> 1) + k;
  digit_stride >>= 1;
#pragma unroll
  for (int p = 0; p < S; ++p) {
    if (EMBED) {
      d[0] = __byte_perm(fr[p], fi[p] ^ 0x80000000u, 0x7632);
      d[Kp >> 1] = __byte_perm(fi[p], fr[p], 0x7632);
    } else {
      d[0] = __byte_perm(fr[p], fi[p], 0x7632);
    }
    d += digit_stride;
  }
}

// Digits of 8 rows by one block, in two passes over K (the largest magnitude,
// then the digits; the second pass finds the rows in L1 or L2).  Rows whose
// entries are contiguous along K go to one warp each; rows that are adjacent
// in memory (element (r+1, k) beside (r, k)) are read 8 rows x 16 bytes at a
// time and turned through shared memory, so that both kinds read whole sectors
// and write 128-byte runs.  (One warp per row reading a column with stride took 34 us
// for the 256 columns of 1280 entries of a chi = 256 H_eff.)
template <bool EMBED, bool SCALED>
__device__ void cut_rows(const Operand& o, int blk, int K, int Kp) {
  __shared__ unsigned long long smax[8][CR];
  __shared__ cplx tile[CR][129];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int per = (o.rows + CR - 1) / CR;
  const int b = blk / per, r0 = (blk - b * per) * CR;
  const cplx* base = o.p + (long long)b * o.sb;
  const long long digit_stride = (long long)o.nb * o.rows * (EMBED ? 2 : 1) * Kp;
  const int r = r0 + w;
  const long long row = ((long long)b * o.rows + r) * (EMBED ? 2 : 1);
  const int Kc = Kp >> 1;
  if (o.sk == 1 || o.sr != 1) {
    if (r >= o.rows) return;
    const cplx* x = base + (long long)r * o.sr;
    unsigned long long mx = 0;
#pragma unroll 4
    for (int k = lane; k < K; k += 32) {
      const cplx v = entry<SCALED>(o, x, k);
      mx = max(mx, max(mag_bits(v.x), mag_bits(v.y)));
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, s));
    const int e = scale_exponent(mx);
    if (lane == 0) o.e[b * o.rows + r] = e;
    for (int k = lane; k < Kc; k += 32)
      write_digits<EMBED>(o, row, digit_stride, Kp, k,
                          k < K ? entry<SCALED>(o, x, k) : cmake(0.0, 0.0), e);
    return;
  }
  const int tr = tid & (CR - 1), tk = tid / CR;              // 32 entries of K at a time
  const bool in = r0 + tr < o.rows;
  const cplx* x = base + (r0 + tr);
  unsigned long long mx = 0;
  if (in) {
#pragma unroll 4
    for (int k = tk; k < K; k += 32) {
      const cplx v = entry<SCALED>(o, x, k);
      mx = max(mx, max(mag_bits(v.x), mag_bits(v.y)));
    }
  }
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
  if (lane < CR) smax[w][lane] = mx;
  __syncthreads();
  mx = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) mx = max(mx, smax[i][w]);
  const int e = scale_exponent(mx);
  if (lane == 0 && r < o.rows) o.e[b * o.rows + r] = e;
  for (int k0 = 0; k0 < Kc; k0 += 128) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = k0 + tk + 32 * i;
      tile[tr][tk + 32 * i] = in && k < K ? entry<SCALED>(o, x, k) : cmake(0.0, 0.0);
    }
    __syncthreads();
    if (r < o.rows) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = k0 + lane + 32 * i;
        if (k < Kc) write_digits<EMBED>(o, row, digit_stride, Kp, k, tile[w][lane + 32 * i], e);
      }
    }
  }
}

template <bool SCALED>
__global__ void __launch_bounds__(256)
k_cut_digits(Operand A, Operand B, int K, int Kp, int blocksA, const int* run_if) {
  if (run_if && *run_if == 0) return;
  if ((int)blockIdx.x < blocksA) cut_rows<true, SCALED>(A, blockIdx.x, K, Kp);
  else cut_rows<false, SCALED>(B, blockIdx.x - blocksA, K, Kp);
}

long long padded_k(int K) { return ((2LL * (K > 0 ? K : 1) + BK - 1) / BK) * BK; }

template <int BN>
cudaError_t launch(const CUtensorMap& ma, const CUtensorMap& mb, EmuShape g, int batch, int sms,
                   cudaStream_t st) {
  typedef Tile<BN> T;
  // the shared-memory attribute is per device; setting it twice from two
  // threads is harmless
  static std::atomic<unsigned long long> attr_done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(attr_done.load() & bit)) {
    e = cudaFuncSetAttribute(k_zgemm_slices<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)T::SMEM);
    if (e != cudaSuccess) return e;
    attr_done.fetch_or(bit);
  }
  g.mt = (g.Mr + BM - 1) / BM;
  g.nt = (g.N + BN - 1) / BN;
  const long long tiles = (long long)g.mt * g.nt * batch;
  if (tiles > (1LL << 30)) return cudaErrorInvalidValue;
  g.tiles = (int)tiles;
  count_launches(1);
  k_zgemm_slices<BN><<<(int)(tiles < sms ? tiles : sms), T::THREADS, T::SMEM, st>>>(ma, mb, g);
  return cudaGetLastError();
}

}  // namespace

// tensor map over (k, row, batch entry, digit) of digit matrices, box
// (32, box_rows, 1, digits), 64-byte swizzle
cudaError_t make_digit_map(CUtensorMap* map, const void* base, long long rows, long long cols,
                           int batch, int digits, int box_rows);

size_t zgemm_emu_scratch_bytes(int M, int N, int K, int batchA, int batchB) {
  return (size_t)S * (2LL * M * batchA + (long long)N * batchB) * padded_k(K) * 2 +
         ((size_t)M * batchA + (size_t)N * batchB) * sizeof(int) + 1024;
}

bool zgemm_emu_rows_fit(int M, int N, int batchA, int batchB) {
  return 2LL * S * M * batchA <= (1LL << 31) && (long long)S * N * batchB <= (1LL << 31);
}

cudaError_t zgemm_emu(const GemmArgs& g, void* scratch, size_t scratch_bytes, int* err,
                      cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
  const int nbA = g.sAb != 0 ? g.batch : 1, nbB = g.sBb != 0 ? g.batch : 1;
  if (scratch_bytes < zgemm_emu_scratch_bytes(g.M, g.N, g.K, nbA, nbB)) return cudaErrorInvalidValue;
  const long long Kp = padded_k(g.K);
  const long long Mr = 2LL * g.M;
  if (!zgemm_emu_rows_fit(g.M, g.N, nbA, nbB)) return cudaErrorInvalidValue;
  __nv_bfloat16* As = reinterpret_cast<__nv_bfloat16*>(scratch);
  __nv_bfloat16* Bs = As + (size_t)S * Mr * nbA * Kp;
  int* eA = reinterpret_cast<int*>(Bs + (size_t)S * g.N * nbB * Kp);
  int* eB = eA + (size_t)g.M * nbA;
  int sms = 0;
  cudaError_t e = device_sms(&sms);
  if (e != cudaSuccess) return e;
  const Operand oA = {g.A, g.sAm, g.sAk, g.sAb, g.conjA ? 1 : 0, g.M, nbA, As, eA,
                      g.kexp, 1};
  const Operand oB = {g.B, g.sBn, g.sBk, g.sBb, g.conjB ? 1 : 0, g.N, nbB, Bs, eB,
                      g.kexp, -1};
  const int blocksA = (g.M + CR - 1) / CR * nbA, blocksB = (g.N + CR - 1) / CR * nbB;
  count_launches(1);
  if (g.kexp)
    k_cut_digits<true><<<blocksA + blocksB, 256, 0, st>>>(oA, oB, g.K, (int)Kp, blocksA, g.run_if);
  else
    k_cut_digits<false><<<blocksA + blocksB, 256, 0, st>>>(oA, oB, g.K, (int)Kp, blocksA, g.run_if);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  EmuShape s;
  s.Mr = (int)Mr; s.N = g.N; s.nkb = (int)(Kp / BK);
  s.a_batched = nbA > 1; s.b_batched = nbB > 1;
  s.ldc = g.ldc; s.sCb = g.sCb;
  s.alpha = g.alpha; s.beta = g.beta; s.gamma = g.gamma;
  s.C = g.C; s.Z = g.Z; s.eA = eA; s.eB = eB; s.run_if = g.run_if; s.err = err;
  // 64 columns per tile when that still gives every SM a tile
  const bool wide = ((Mr + BM - 1) / BM) * ((g.N + 63) / 64) * (long long)g.batch >= sms;
  CUtensorMap ma, mb;
  e = make_digit_map(&ma, As, Mr, Kp, nbA, S, BM);
  if (e != cudaSuccess) return e;
  e = make_digit_map(&mb, Bs, g.N, Kp, nbB, S, wide ? 64 : 32);
  if (e != cudaSuccess) return e;
  return wide ? launch<64>(ma, mb, s, g.batch, sms, st) : launch<32>(ma, mb, s, g.batch, sms, st);
}

}  // namespace ite
