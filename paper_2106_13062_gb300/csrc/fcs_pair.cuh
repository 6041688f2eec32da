// fcs_pair.cuh -- the forward real FFT of the CP route for P = 1024 NR,
// NR = 16 or 32 (M = 512 NR complex points), on packed FP32 arithmetic.
//
// The transform is a decimation in time over NR rows of 512 points,
//   Z[k + 512 q1] = sum_w W_NR^(w q1) W_M^(w k) Y_w[k],  Y_w = FFT_512(z[NR m + w]).
// Blackwell's packed FP32 instructions (add/mul/fma.f32x2) do two
// operations per issue slot and lane pair; a plain FP32 stream runs out of
// issue slots (the loads, stores and moves of an FFT compete with it) long
// before the FP32 pipe is full.  So rows are processed in pairs: a C2 holds the same element
// of rows 2k and 2k+1, every operation of a row FFT is one packed operation on
// both, and one 16-byte shared access moves both.  In the column step the
// packed halves are the even and the odd rows, whose NR/2-point DFTs run in
// lockstep; only the last radix-2 stage of the column crosses the halves.
//
// Row step (one warp, one row pair).  Lane (s, e) = (lane / 2, lane mod 2)
// takes the outputs k = 2 k' + e:
//   g[m] = (z[m] + (-1)^e z[m + 256]) W512^(e m),  Y[2 k' + e] = FFT_256(g)[k'],
// and FFT_256 is 16 x 16 with one transpose among the lanes of equal e.  The second
// half of a row is empty unless a hash range exceeds P / 2, so the input
// radix-2 usually costs nothing, and no value is read twice (a radix-2 step
// after the transpose has both half-warps read all of it).
//
// Column step: thread t owns the columns u and 512 - u (u = t + 1 + NT c, so u
// = 1 .. 256), so every pair (q, M - q) of the real-FFT unpack lies in one
// thread, without shuffles, and the second column's twiddles are the
// conjugates of the first's.  (u = 256 pairs with itself: its second half
// repeats the first.)  Column 0 holds the NR + 1 bins X[512 i], the real FFT of
// the 2 NR row sums, which one warp evaluates directly, one bin per lane:
// no thread of the column step is an exception.
//
// A rank's running mode product and the rank sum (64 words each per thread,
// 128 at NR = 32) live in tensor memory: they are touched once per transform,
// and without them a thread's 32 spectrum values and the temporaries fit 128
// registers, so two 256-thread CTAs share an SM at NR = 16 and one's barriers
// hide behind the other.
#pragma once

#include "fcs_fft.cuh"

namespace fcs {
namespace pfft {

// ---------------------------------------------------------------- packed FP32
struct f2x {
  unsigned long long v;
};
__device__ __forceinline__ f2x pk(float lo, float hi) {
  f2x r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float lo(f2x a) {
  float x, y;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
  return x;
}
__device__ __forceinline__ float hi(f2x a) {
  float x, y;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
  return y;
}
__device__ __forceinline__ f2x splat(float x) { return pk(x, x); }
__device__ __forceinline__ f2x add2(f2x a, f2x b) {
  f2x r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2x mul2(f2x a, f2x b) {
  f2x r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2x fma2(f2x a, f2x b, f2x c) {
  f2x r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ f2x neg2(f2x a) { return pk(-lo(a), -hi(a)); }
__device__ __forceinline__ f2x sub2(f2x a, f2x b) { return fma2(b, splat(-1.f), a); }

// Two complex numbers.
struct C2 {
  f2x re{0ull}, im{0ull};
};
__device__ __forceinline__ C2 make_c2(float4 x) { return C2{pk(x.x, x.y), pk(x.z, x.w)}; }
__device__ __forceinline__ float4 c2_float4(C2 a) {
  return make_float4(lo(a.re), hi(a.re), lo(a.im), hi(a.im));
}
__device__ __forceinline__ C2 cadd(C2 a, C2 b) { return C2{add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 csub(C2 a, C2 b) { return C2{sub2(a.re, b.re), sub2(a.im, b.im)}; }
__device__ __forceinline__ void bfly_mi(C2 a, C2 b, C2 &x, C2 &y) {
  x = C2{add2(a.re, b.im), sub2(a.im, b.re)};
  y = C2{sub2(a.re, b.im), add2(a.im, b.re)};
}
// a * w with w given as (re, im, -im).
__device__ __forceinline__ C2 cmul3(C2 a, f2x wr, f2x wi, f2x nwi) {
  return C2{fma2(a.re, wr, mul2(a.im, nwi)), fma2(a.re, wi, mul2(a.im, wr))};
}
// Both numbers times the same w.
__device__ __forceinline__ C2 cmul_same(C2 a, float2 w) {
  return cmul3(a, splat(w.x), splat(w.y), splat(-w.y));
}
__device__ __forceinline__ C2 cmul(C2 a, C2 w) { return cmul3(a, w.re, w.im, neg2(w.im)); }
// bfly_tw of fcs_internal.cuh on both numbers.
template <int J>
__device__ __forceinline__ void bfly_tw(C2 &a, C2 &b) {
  static_assert(J > 0 && J < 32 && J != 16, "twiddle index");
  f2x ux, uy;
  if constexpr (J <= 8 || J >= 24) {
    constexpr float t = J <= 8 ? tan64_q(J) : -tan64_q(32 - J);     // s / c
    constexpr float f = cos64(J);
    ux = fma2(splat(t), b.im, b.re);
    uy = fma2(splat(-t), b.re, b.im);
    const C2 a0 = a;
    a = C2{fma2(splat(f), ux, a0.re), fma2(splat(f), uy, a0.im)};
    b = C2{fma2(splat(-f), ux, a0.re), fma2(splat(-f), uy, a0.im)};
  } else {
    constexpr float k = J <= 16 ? tan64_q(16 - J) : -tan64_q(J - 16);   // c / s
    constexpr float f = sin64(J);
    ux = fma2(splat(k), b.re, b.im);
    uy = fma2(splat(-k), b.im, b.re);                  // minus the imaginary part
    const C2 a0 = a;
    a = C2{fma2(splat(f), ux, a0.re), fma2(splat(-f), uy, a0.im)};
    b = C2{fma2(splat(-f), ux, a0.re), fma2(splat(f), uy, a0.im)};
  }
}

// ---------------------------------------------------------------- geometry
__host__ __device__ constexpr int log2_const(int n) { return n <= 1 ? 0 : 1 + log2_const(n / 2); }

template <int NR>
struct Geo {
  static constexpr int LNR = log2_const(NR);
  static constexpr int M = 512 * NR;
  static constexpr int LM = 9 + LNR;                  // log2 M
  static_assert(NR == 16 || NR == 32, "P = 16384 or 32768");
  static constexpr int NT = 256;                      // threads per CTA
  static constexpr int CTAS = NR == 16 ? 2 : 1;       // CTAs per SM
  static constexpr int WARPS = NT / 32;
  static constexpr int RPW = NR / 2 / WARPS;          // row pairs per warp
  static constexpr int NCP = 256 / NT;                // column pairs per thread
  static constexpr int H = NR / 2;
  // the row step's transpose: padded rows at NR = 32, swizzled ones where the
  // shared memory decides how many blocks share an SM
  static constexpr bool PAD = NR == 32;
  static constexpr int RS = PAD ? 549 : 513;          // row-pair stride of B (float4)
  static constexpr int WPT = NCP * 4 * NR;            // words per thread of one spectrum
  static constexpr int TCOLS = 2 * WPT * (WARPS / 4); // tensor-memory columns per CTA
};

// Shared-memory layout: B (row pairs) | input twiddles | transpose twiddles |
// column-step twiddles | column-0 twiddles | scatter buffer (row pairs of ra
// float4).
template <int NR>
struct Smem {
  using G = Geo<NR>;
  static constexpr size_t kB = 0;
  static constexpr size_t kT0 = kB + sizeof(float4) * (NR / 2) * G::RS;
  static constexpr size_t kT1 = kT0 + sizeof(float2) * 16 * 32;
  static constexpr size_t kT2 = kT1 + sizeof(float2) * 15 * 16;
  static constexpr size_t kT3 = kT2 + sizeof(float2) * 256 * (G::LNR + 1);
  static constexpr size_t kA = kT3 + sizeof(float2) * 2 * NR;
  static constexpr size_t bytes(int ra) { return kA + sizeof(float4) * (NR / 2) * size_t(ra); }
};

// Blocks that share an SM with `smem` bytes of dynamic shared memory each
// (228 KiB per SM; 1 KiB reserved and some static arrays per block).  The
// runtime's occupancy query answers 1 for any kernel that allocates tensor
// memory.
template <int NR>
int blocks_per_sm(size_t smem) {
  const int n = int(size_t(233472) / (smem + 1024 + 256));
  return n < 1 ? 1 : n < Geo<NR>::CTAS ? n : Geo<NR>::CTAS;
}

static_assert(Smem<32>::bytes((kPair32MaxJ + 63) / 64) <= 232448 - 1024, "scatter buffer fits");

// Float index of real sample h in the scatter buffer (z[m], m = h / 2, is
// element m / NR of row m mod NR; rows 2k and 2k+1 are interleaved).
template <int NR>
__device__ __forceinline__ int a_index(int h, int ra) {
  const int m = h >> 1, w = m & (NR - 1);
  return (((w >> 1) * ra + (m / NR)) << 2) + ((h & 1) << 1) + (w & 1);
}
// Float index of the real part of z[m] in B (imaginary part two further on).
template <int NR>
__device__ __forceinline__ int b_index(int m) {
  const int w = m & (NR - 1);
  return (((w >> 1) * Geo<NR>::RS + (m / NR)) << 2) + (w & 1);
}

// Twiddle tables from tw[k] = exp(-2 pi i k / 2^15):
//   t0[r*32 + lane] = W512^(e (s + 16 r)), t1[(ka - 1)*16 + s] = W256^(s ka),
//   t2[b*256 + u - 1] = W_M^(u 2^b) (b < log2 NR), t2[LNR*256 + u - 1] = W_P^u,
//   t3[k] = exp(-2 pi i k / (2 NR)).
template <int NR>
__device__ __forceinline__ void fill_twiddles(unsigned char *smem, const float2 *__restrict__ tw) {
  using G = Geo<NR>;
  float2 *t0 = reinterpret_cast<float2 *>(smem + Smem<NR>::kT0);
  float2 *t1 = reinterpret_cast<float2 *>(smem + Smem<NR>::kT1);
  float2 *t2 = reinterpret_cast<float2 *>(smem + Smem<NR>::kT2);
  for (int k = threadIdx.x; k < 512; k += G::NT)
    t0[k] = k & 1 ? __ldg(&tw[(((k & 31) >> 1) + 16 * (k >> 5)) << 6]) : make_float2(1.f, 0.f);
  for (int k = threadIdx.x; k < 240; k += G::NT) t1[k] = __ldg(&tw[((k & 15) * (1 + (k >> 4))) << 7]);
#pragma unroll
  for (int c = 0; c < G::NCP; ++c) {
    const int t = threadIdx.x + c * G::NT, u = t + 1;
#pragma unroll
    for (int b = 0; b < G::LNR; ++b) t2[b * 256 + t] = __ldg(&tw[(u << b) << (kLogTwN - G::LM)]);
    t2[G::LNR * 256 + t] = __ldg(&tw[u << (kLogTwN - G::LM - 1)]);
  }
  if (threadIdx.x < 2 * NR)
    reinterpret_cast<float2 *>(smem + Smem<NR>::kT3)[threadIdx.x] =
        __ldg(&tw[threadIdx.x << (kLogTwN - G::LNR - 1)]);
}

// ---------------------------------------------------------------- tensor memory
// Each thread owns 2 WPT words of its warp's lane quadrant.
template <int NR>
__device__ __forceinline__ uint32_t tmem_alloc(uint32_t *slot) {
  if (threadIdx.x < 32) {
    const uint32_t a = uint32_t(__cvta_generic_to_shared(slot));
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(a),
                 "n"(Geo<NR>::TCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return *slot;
}
// After every thread's last tensor-memory access (which it has waited for).
template <int NR>
__device__ __forceinline__ void tmem_free(uint32_t base) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base),
                 "n"(Geo<NR>::TCOLS)
                 : "memory");
}
// This thread's words start here.
template <int NR>
__device__ __forceinline__ uint32_t tmem_mine(uint32_t base) {
  const uint32_t w = threadIdx.x >> 5;
  return base + ((w & 3) << 21) + (w >> 2) * (2 * Geo<NR>::WPT);
}
struct Tm16 {
  uint32_t r[16];
};
__device__ __forceinline__ void tmem_st16(uint32_t addr, const Tm16 &x) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16};" ::"r"(addr),
      "r"(x.r[0]), "r"(x.r[1]), "r"(x.r[2]), "r"(x.r[3]), "r"(x.r[4]), "r"(x.r[5]), "r"(x.r[6]),
      "r"(x.r[7]), "r"(x.r[8]), "r"(x.r[9]), "r"(x.r[10]), "r"(x.r[11]), "r"(x.r[12]),
      "r"(x.r[13]), "r"(x.r[14]), "r"(x.r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, Tm16 &x) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];"
      : "=r"(x.r[0]), "=r"(x.r[1]), "=r"(x.r[2]), "=r"(x.r[3]), "=r"(x.r[4]), "=r"(x.r[5]),
        "=r"(x.r[6]), "=r"(x.r[7]), "=r"(x.r[8]), "=r"(x.r[9]), "=r"(x.r[10]), "=r"(x.r[11]),
        "=r"(x.r[12]), "=r"(x.r[13]), "=r"(x.r[14]), "=r"(x.r[15])
      : "r"(addr)
      : "memory");
}
// The loaded registers are operands, so that no use moves above the wait.
__device__ __forceinline__ void tmem_wait_ld(Tm16 &x) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(x.r[0]), "+r"(x.r[1]), "+r"(x.r[2]), "+r"(x.r[3]), "+r"(x.r[4]),
                 "+r"(x.r[5]), "+r"(x.r[6]), "+r"(x.r[7]), "+r"(x.r[8]), "+r"(x.r[9]),
                 "+r"(x.r[10]), "+r"(x.r[11]), "+r"(x.r[12]), "+r"(x.r[13]), "+r"(x.r[14]),
                 "+r"(x.r[15])::"memory");
}
__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ C2 tm_get(const Tm16 &x, int i) {
  return C2{pk(__uint_as_float(x.r[4 * i]), __uint_as_float(x.r[4 * i + 1])),
            pk(__uint_as_float(x.r[4 * i + 2]), __uint_as_float(x.r[4 * i + 3]))};
}
__device__ __forceinline__ void tm_set(Tm16 &x, int i, C2 c) {
  x.r[4 * i] = __float_as_uint(lo(c.re));
  x.r[4 * i + 1] = __float_as_uint(hi(c.re));
  x.r[4 * i + 2] = __float_as_uint(lo(c.im));
  x.r[4 * i + 3] = __float_as_uint(hi(c.im));
}

// ---------------------------------------------------------------- row step
// The 512-point FFTs of K row pairs (K = 2: both at once, for a warp that has
// two and the registers for them): `in` (ra <= 512 elements, the rest zero) to
// `out` (512 elements, with PAD 548, also the transpose scratch); the second
// pair `ink`, `outk` further on.  NZ: number of 16-element blocks of the first
// half-row that can be non-zero (ra <= 16 NZ <= 256), 32 = the whole row.
// INPLACE: in == out; otherwise `in` is cleared.
template <int NZ, bool INPLACE, int K, bool PAD>
__device__ __forceinline__ void row_step(float4 *in, int ink, int ra, float4 *out, int outk,
                                         const float2 *t0, const float2 *t1) {
  constexpr int NB = NZ > 16 ? 16 : NZ;
  const int l = threadIdx.x & 31, s = l >> 1, e = l & 1;
  C2 v[K][16];
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int r = 0; r < NB; ++r) {
      const float4 *x = in + k * ink;
      const int m = s + 16 * r;
      v[k][r] = make_c2(m < ra ? x[m] : make_float4(0.f, 0.f, 0.f, 0.f));
      if constexpr (NZ > 16) {
        const C2 y = make_c2(m + 256 < ra ? x[m + 256] : make_float4(0.f, 0.f, 0.f, 0.f));
        const f2x sg = splat(e ? -1.f : 1.f);
        v[k][r] = C2{fma2(y.re, sg, v[k][r].re), fma2(y.im, sg, v[k][r].im)};
      }
    }
  __syncwarp();
  if constexpr (!INPLACE) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      for (int i = l; i < ra; i += 32) in[k * ink + i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
#pragma unroll
  for (int r = 0; r < NB; ++r) {
    const float2 w = t0[r * 32 + l];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k][r] = cmul_same(v[k][r], w);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) DftNZ<16, NB>::run(v[k]);
#pragma unroll
  for (int ka = 1; ka < 16; ++ka) {
    const float2 w = t1[(ka - 1) * 16 + s];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k][ka] = cmul_same(v[k][ka], w);
  }
  // transpose in place of the result; the eight lanes of an access phase
  // (four s, two e) use distinct 16-byte banks both ways: rows of 17 and the
  // odd lanes' part 276 (4 mod 8) further on, or element ka of lane (s, e) at
  // column ka ^ (s mod 8) ^ 4 e of a row of 16
  float4 *T = out + e * (PAD ? 276 : 256);
  const int e4 = e << 2;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int ka = 0; ka < 16; ++ka)
      T[k * outk + (PAD ? s * 17 + ka : s * 16 + (ka ^ (s & 7) ^ e4))] = c2_float4(v[k][ka]);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int q = 0; q < 16; ++q)
      v[k][q] = make_c2(T[k * outk + (PAD ? q * 17 + s : q * 16 + (s ^ (q & 7) ^ e4))]);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < K; ++k) Dft<16>::run(v[k]);
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int q = 0; q < 16; ++q) out[k * outk + 2 * s + e + 32 * q] = c2_float4(v[k][q]);
}

// row_step of scatter-buffer row pairs with the input pruning that fits their
// height: 8, 11, 16 or all 32 blocks of 16.  Equal hash lengths J in order 3
// give ra in (85, 171], in order 4 (64, 128]; one long mode gives up to 512.
// ra is the same for the whole block, so the branch is uniform.
template <int K, bool PAD>
__device__ __forceinline__ void scatter_row_step(float4 *in, int ink, int ra, float4 *out,
                                                 int outk, const float2 *t0, const float2 *t1) {
  if (ra <= 128)
    row_step<8, false, K, PAD>(in, ink, ra, out, outk, t0, t1);
  else if (ra <= 176)
    row_step<11, false, K, PAD>(in, ink, ra, out, outk, t0, t1);
  else if (ra <= 256)
    row_step<16, false, K, PAD>(in, ink, ra, out, outk, t0, t1);
  else
    row_step<32, false, K, PAD>(in, ink, ra, out, outk, t0, t1);
}

// ---------------------------------------------------------------- column step
// Last radix-2 stage of a column: x holds element K of the even and of the
// odd rows' DFTs; y0, y1 are elements K and K + NR/2 of the column's DFT.
template <int NR, int K>
__device__ __forceinline__ void combine(C2 x, float2 &y0, float2 &y1) {
  float2 a = make_float2(lo(x.re), lo(x.im)), b = make_float2(hi(x.re), hi(x.im));
  if constexpr (K == 0) {
    y0 = fcs::cadd(a, b);
    y1 = fcs::csub(a, b);
  } else if constexpr (4 * K == NR) {
    fcs::bfly_mi(a, b, y0, y1);
  } else {
    fcs::bfly_tw<K *(64 / NR)>(a, b);
    y0 = a;
    y1 = b;
  }
}
template <int NR, int K, bool SWAP>
__device__ __forceinline__ void combine_all(C2 *x) {
  if constexpr (K < NR / 2) {
    float2 a, b;
    combine<NR, K>(x[K], a, b);
    if constexpr (SWAP && K > 0)
      x[K] = C2{pk(b.x, a.x), pk(b.y, a.y)};
    else
      x[K] = C2{pk(a.x, b.x), pk(a.y, b.y)};
    combine_all<NR, K + 1, SWAP>(x);
  }
}

// P[k] = (w^(2k), w^(2k+1)) for k < 2^(LNR-1) from P[0] and w[b] = w^(2^b).
template <int LNR, int B = 1>
__device__ __forceinline__ void pair_powers(C2 *P, const float2 *w) {
  if constexpr (B < LNR) {
    constexpr int n = 1 << (B - 1);
#pragma unroll
    for (int k = 0; k < n; ++k) P[k + n] = cmul_same(P[k], w[B]);
    pair_powers<LNR, B + 1>(P, w);
  }
}

// Columns u = threadIdx.x + 1 + c NT and 512 - u up to the complex spectrum:
//   xa[K] = (A[K], A[K + H]),  A[q1] = Z[u + 512 q1], H = NR / 2,
//   xc[0] = (C[0], C[H]), xc[K] = (C[K + H], C[K]) for K > 0,
//   C[(q1 + 1) mod NR] = Z[512 - u + 512 q1]
// (the second column's twiddles are the conjugates of the first's, which
// rotates its DFT's output by one).  HALF: all of it times 1/2, by the first
// twiddles.
template <int NR, bool HALF = false>
__device__ __forceinline__ void column_step(const float4 *B, const float2 *t2, int c, C2 *xa,
                                            C2 *xc) {
  using G = Geo<NR>;
  const int t = threadIdx.x + c * G::NT;
#pragma unroll
  for (int k = 0; k < G::H; ++k) {
    xa[k] = make_c2(B[k * G::RS + t + 1]);
    xc[k] = make_c2(B[k * G::RS + 511 - t]);
  }
  // W^(2k), W^(2k+1) for row pair k: products of at most log2 NR factors
  float2 w[G::LNR];
#pragma unroll
  for (int b = 0; b < G::LNR; ++b) w[b] = t2[b * 256 + t];
  C2 P[G::H];
  constexpr float f = HALF ? 0.5f : 1.f;
  P[0] = C2{pk(f, f * w[0].x), pk(0.f, f * w[0].y)};
  pair_powers<G::LNR>(P, w);
#pragma unroll
  for (int k = 0; k < G::H; ++k) {
    const f2x ni = neg2(P[k].im);
    xa[k] = cmul3(xa[k], P[k].re, P[k].im, ni);
    xc[k] = cmul3(xc[k], P[k].re, ni, P[k].im);
  }
  Dft<G::H>::run(xa);
  Dft<G::H>::run(xc);
  combine_all<NR, 0, false>(xa);
  combine_all<NR, 0, true>(xc);
}

// Real-FFT unpack of the column pair, in place: xa[K] holds TWICE X[q] and
// xc[(H - K) mod H] TWICE X[M - q] for q = u + 512 K (low half) and
// u + 512 (K + H) (high half); X[q] and X[M - q] themselves after a column
// step with HALF.
template <int NR>
__device__ __forceinline__ void unpack(const float2 *t2, int c, C2 *xa, C2 *xc) {
  using G = Geo<NR>;
  constexpr int H = G::H;
  const float2 wP = t2[G::LNR * 256 + threadIdx.x + c * G::NT];
#pragma unroll
  for (int K = 0; K < H; ++K) {
    const C2 za = xa[K], zb = xc[(H - K) % H];
    // W_P^(u + 512 K) and, W_P^(512 H) being -i, W_P^(u + 512 (K + H))
    const float2 w0 = K == 0 ? wP : fcs::cmul(wP, unit64(K * 32 / NR));
    const f2x er = add2(za.re, zb.re), ei = sub2(za.im, zb.im);
    const f2x orr = add2(za.im, zb.im), oi = sub2(zb.re, za.re);
    const f2x wr = pk(w0.x, w0.y), wi = pk(w0.y, -w0.x), nwi = pk(-w0.y, w0.x);
    const f2x tr = fma2(wr, orr, mul2(nwi, oi)), ti = fma2(wr, oi, mul2(wi, orr));
    xa[K] = C2{add2(er, tr), add2(ei, ti)};
    xc[(H - K) % H] = C2{sub2(er, tr), sub2(ti, ei)};
  }
}

// Bin of the value in xa (b = 0) or xc[(H - K) mod H] (b = 1), half `half`.
template <int NR>
__device__ __forceinline__ int bin_of(int c, int b, int K, int half) {
  using G = Geo<NR>;
  const int q = threadIdx.x + 1 + c * G::NT + 512 * (K + half * G::H);
  return b == 0 ? q : G::M - q;
}

// Column 0, by one whole warp: lane i < NR returns TWICE X[512 i], lane 0 the
// packed real bins (2 X[0], 2 X[M]).  With y[2w + c] the real (c = 0) and
// imaginary part of Y_w[0], X[512 i] = sum_j y[j] exp(-2 pi i i j / (2 NR)).
// The 32 / NR lanes of a bin share the sum.
template <int NR>
__device__ __forceinline__ float2 column0(const float4 *B, const float2 *t3) {
  using G = Geo<NR>;
  constexpr int S = 32 / NR;
  const int l = threadIdx.x & 31, i = l & (NR - 1), sub = l / NR;
  float2 x = make_float2(0.f, 0.f);
#pragma unroll
  for (int kk = 0; kk < G::H / S; ++kk) {
    const int k = kk * S + sub;
    const float4 v = B[k * G::RS];                     // rows 2k and 2k + 1
    const float y[4] = {v.x, v.z, v.y, v.w};           // samples 4k .. 4k + 3
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float2 w = t3[(i * (4 * k + j)) & (2 * NR - 1)];
      if (i == 0) w.y = (j & 1) ? -1.f : 1.f;          // (-1)^j: bin M
      x.x = fmaf(y[j], w.x, x.x);
      x.y = fmaf(y[j], w.y, x.y);
    }
  }
#pragma unroll
  for (int o = NR; o < 32; o <<= 1) {
    x.x += __shfl_xor_sync(0xffffffffu, x.x, o);
    x.y += __shfl_xor_sync(0xffffffffu, x.y, o);
  }
  return make_float2(2.f * x.x, 2.f * x.y);
}

// The complex spectrum's column 0 of a packed transform, by one whole warp:
// lane i < NR returns Z[512 i] = sum_w Y_w[0] exp(-2 pi i i w / NR).
template <int NR>
__device__ __forceinline__ float2 column0_complex(const float4 *B, const float2 *t3) {
  using G = Geo<NR>;
  const int i = threadIdx.x & (NR - 1);
  float2 x = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int w = 0; w < NR; ++w) {
    const float *p = reinterpret_cast<const float *>(B + (w >> 1) * G::RS) + (w & 1);
    const float2 z = fcs::cmul(make_float2(p[0], p[2]), t3[(2 * i * w) & (2 * NR - 1)]);
    x = fcs::cadd(x, z);
  }
  return x;
}

}  // namespace pfft
}  // namespace fcs
