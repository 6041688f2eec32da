// fcs_dit.cuh -- the forward real FFT of the CP route for P = 8192 (M = 4096
// complex points) on 256 threads.
//
// Decimation in time splits z into the 8 sub-sequences z_w[m2] = z[8 m2 + w]:
//   Z[k + 512 q1] = sum_w W8^(w q1) W_M^(w k) Y_w[k],   Y_w = FFT_512(z_w).
// Step 1 (warp-local): warp w computes Y_w, 16 values per lane, as
//   Y_w[ka + 16 kb] = sum_l W32^(l kb) W512^(l ka) sum_r W16^(r ka) z_w[l + 32 r]:
//   a radix-16 DFT over r in registers (input-pruned: rows r >= RMAX of the
//   scatter buffer are empty), the twiddle W512^(l ka), a transpose through
//   a warp-private stretch of B (__syncwarp only), then the 16 32-point DFTs
//   over l split between the two half-warps (half e takes the outputs
//   kb = 2 kk + e after one radix-2 step); Y_w goes to row w of B.
// Step 2 (after one block barrier): thread t takes the two columns ua(t) and
//   ub(t) = 512 - ua(t) (t = 0: columns 256 and 0), twiddles each by
//   W_M^(w q2), takes two 8-point DFTs, and does the real-FFT unpack inside
//   the thread: bin ua + 512 q1 pairs with ub + 512 (7 - q1).
// The row-pair engine of fcs_pair.cuh, which takes over at P = 16384, has only
// four warps with a row pair here, and a chain of its transforms is longer:
// order 3, I = 300 per call 19.7 us for 15.3 at R = 8, D = 5 and 54.5 for 48.7 at
// R = 100, D = 10; order 2, I = 1500 25 for 16 and 58.6 for 45.
#pragma once

#include "fcs_fft.cuh"

namespace fcs {
namespace wdit {

constexpr int kRS = 576;     // row stride of B (float2)
constexpr int kTR = 18;      // row stride of the step-1 transpose (float2, even: 16-byte pairs)
static_assert(31 * kTR + 16 <= kRS, "transpose fits in one row of B");

// Twice the real-FFT unpack of one pair: with w = W_P^q,
// 2 X[q] = 2E + w 2O and 2 X[M - q] = conj(2E - w 2O).
__device__ __forceinline__ void unpack2_twice(float2 za, float2 zb, float2 w, float2 &xa,
                                              float2 &xb) {
  const float2 e = make_float2(za.x + zb.x, za.y - zb.y);
  const float2 o = make_float2(za.y + zb.y, zb.x - za.x);
  const float2 t = cmul(w, o);
  xa = cadd(e, t);
  xb = cconj(csub(e, t));
}

// Step 1 for row w: the 512-point FFT of in_row (ra float2 entries; with SWZ
// column c of row w sits at c ^ w) into out_row (kRS float2, also the
// transpose scratch).  INPLACE: in_row == out_row, so the warp synchronises
// after reading its input and nothing is cleared; otherwise the entries read
// are cleared.  No block barrier inside.
template <int RMAX, bool SWZ, bool INPLACE>
__device__ __forceinline__ void step1_row(float2 *in_row, int ra, float2 *out_row,
                                          const float2 *tws, int w) {
  const int l = threadIdx.x & 31;
  const int lc = SWZ ? (l ^ w) : l;
  float2 v[16];
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const int m2 = l + 32 * r;
    v[r] = (r < RMAX && m2 < ra) ? in_row[lc + 32 * r] : make_float2(0.f, 0.f);
  }
  if (INPLACE) {
    __syncwarp();
  } else {
#pragma unroll
    for (int r = 0; r < RMAX; ++r) {
      const int m2 = l + 32 * r;
      if (m2 < ra) in_row[lc + 32 * r] = make_float2(0.f, 0.f);
    }
  }
  DftNZ<16, RMAX>::run(v);
#pragma unroll
  for (int ka = 1; ka < 16; ++ka) v[ka] = cmul(v[ka], tws[ka * 32 + l]);   // W512^(l ka)
  float2 *T = out_row;
#pragma unroll
  for (int ka = 0; ka < 16; ka += 2)
    *reinterpret_cast<float4 *>(T + l * kTR + ka) =
        make_float4(v[ka].x, v[ka].y, v[ka + 1].x, v[ka + 1].y);
  __syncwarp();
  const int j = l & 15;
  const bool odd = l >= 16;
  const float sg = odd ? -1.f : 1.f;
#pragma unroll
  for (int lp = 0; lp < 16; ++lp) {
    const float2 a = T[lp * kTR + j], b = T[(lp + 16) * kTR + j];
    float2 g = make_float2(fmaf(sg, b.x, a.x), fmaf(sg, b.y, a.y));
    if (lp > 0) {
      const float2 wv = unit64(2 * lp);
      g = cmul(g, make_float2(odd ? wv.x : 1.f, odd ? wv.y : 0.f));
    }
    v[lp] = g;
  }
  Dft<16>::run(v);
  __syncwarp();
  const int k0 = j + (odd ? 16 : 0);
#pragma unroll
  for (int kk = 0; kk < 16; ++kk) T[k0 + 32 * kk] = v[kk];
}

constexpr int kM = 1 << 12;
constexpr int kNT = 256;
constexpr int kTw2 = 16 * 32;               // after the step-1 table W512^(l ka)
constexpr int kTwLen = kTw2 + 7 * kNT;      // W_M^(ua 2^b), W_M^(ub 2^b) (b < 3), W_P^ua

__device__ __forceinline__ int ua_of(int t) { return t ? t : 256; }
__device__ __forceinline__ int ub_of(int t) { return t ? 512 - t : 0; }

// Float index of real sample h in the 8-row scatter buffer (row m mod 8,
// column m / 8 for m = h / 2; rows of ra float2).
__device__ __forceinline__ int a_index(int h, int ra) {
  const int m = h >> 1;
  return 2 * ((m & 7) * ra + (m >> 3)) + (h & 1);
}

// Position of z[m] in an 8-row buffer of row stride kRS, rows XOR-swizzled
// (row w holds z[8 m2 + w] at column m2 ^ w), read back by
// step1_row<16, true, true>.
__device__ __forceinline__ int row_pos_swz(int m) {
  const int w = m & 7;
  return w * kRS + ((m >> 3) ^ w);
}

// Per-CTA twiddle table: the step-1 part (W512^(l ka) at ka*32 + l), then for
// thread t W_M^(ua 2^b) at kTw2 + b*256 + t, W_M^(ub 2^b) at
// kTw2 + (3 + b)*256 + t (b < 3) and W_P^ua at kTw2 + 6*256 + t, from
// tw[k] = exp(-2 pi i k / 2^15).  Every load is issued before the first store.
__device__ __forceinline__ void fill_twiddles(float2 *tws, const float2 *__restrict__ tw) {
  constexpr int PER = kTwLen / kNT;
  static_assert(kTwLen % kNT == 0, "twiddle table fill");
  float2 v[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int e = threadIdx.x + k * kNT;
    if (e < kTw2) {
      const int ka = e >> 5, l = e & 31;
      v[k] = __ldg(&tw[(l * ka) << (kLogTwN - 9)]);
    } else {
      const int b = (e - kTw2) >> 8, t = (e - kTw2) & (kNT - 1);
      const int ua = ua_of(t), ub = ub_of(t);
      v[k] = b < 3   ? __ldg(&tw[(ua << b) << (kLogTwN - 12)])
             : b < 6 ? __ldg(&tw[(ub << (b - 3)) << (kLogTwN - 12)])
                     : __ldg(&tw[ua << (kLogTwN - 13)]);
    }
  }
#pragma unroll
  for (int k = 0; k < PER; ++k) tws[threadIdx.x + k * kNT] = v[k];
}

// Step 2 up to the complex spectrum: va[q1] = Z[ua + 512 q1],
// vb[q1] = Z[ub + 512 q1].
__device__ __forceinline__ void step2_complex(const float2 *B, const float2 *tws, float2 (&va)[8],
                                              float2 (&vb)[8]) {
  const int t = threadIdx.x;
  const int ua = ua_of(t), ub = ub_of(t);
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    va[w] = B[w * kRS + ua];
    vb[w] = B[w * kRS + ub];
  }
  float2 wa[3], wb[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    wa[b] = tws[kTw2 + b * kNT + t];
    wb[b] = tws[kTw2 + (3 + b) * kNT + t];
  }
  twiddle_powers<3>(va, wa);
  twiddle_powers<3>(vb, wb);
  Dft<8>::run(va);
  Dft<8>::run(vb);
}

// Step 2 with the real-FFT unpack: TWICE the half-spectrum values,
// va[q1] = 2 X[ua + 512 q1], vb[q1] = 2 X[ub + 512 q1]; for thread 0 (ub = 0)
// vb[0] packs the two real bins (2 X[0], 2 X[M]).
__device__ __forceinline__ void step2(const float2 *B, const float2 *tws, float2 (&va)[8],
                                      float2 (&vb)[8]) {
  const int t = threadIdx.x;
  step2_complex(B, tws, va, vb);
  if (t != 0) {
    const float2 wP = tws[kTw2 + 6 * kNT + t];      // W_P^ua, P = 8192
#pragma unroll
    for (int q1 = 0; q1 < 8; ++q1) {
      // W_P^(ua + 512 q1) = W_P^ua exp(-2 pi i q1 / 16); partner ub + 512 (7 - q1)
      const float2 wq = q1 == 0 ? wP : cmul(wP, unit64(4 * q1));
      unpack2_twice(va[q1], vb[7 - q1], wq, va[q1], vb[7 - q1]);
    }
  } else {
    // column 256 pairs with itself: 256 + 512 q1 <-> 256 + 512 (7 - q1)
#pragma unroll
    for (int q1 = 0; q1 < 4; ++q1)
      unpack2_twice(va[q1], va[7 - q1], unit64(2 + 4 * q1), va[q1], va[7 - q1]);
    // column 0: 512 q1 <-> 512 (8 - q1); q1 = 0 and 4 pair with themselves
    const float2 z0 = vb[0], z4 = vb[4];
    vb[0] = make_float2(2.f * (z0.x + z0.y), 2.f * (z0.x - z0.y));
    vb[4] = make_float2(2.f * z4.x, -2.f * z4.y);
#pragma unroll
    for (int q1 = 1; q1 < 4; ++q1) unpack2_twice(vb[q1], vb[8 - q1], unit64(4 * q1), vb[q1], vb[8 - q1]);
  }
}

}  // namespace wdit
}  // namespace fcs
