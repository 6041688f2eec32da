// fcs_cp_run.cuh -- the CP-route work of one (sketch d, rank group), eq.
// (FCS_syn), shared by the single-problem kernels (fcs_cp.cu) and the batch
// kernels (fcs_batch.cu).  For each rank r and mode n the signed factor
// column is count-sketched (Def. 1) into a compact shared buffer (the zero
// padding up to P is never stored), transformed by a block real FFT whose
// output half spectrum stays in registers, and multiplied into the
// per-thread mode product; the product is added into a shared rank
// accumulator, so the rank sum stays in the frequency domain.  The next
// column's factor values and hashes are prefetched into registers while the
// current one is transformed.  The group's partial spectrum then goes into
// the sketch's global accumulator with atomics, and the group that completes
// sketch d (ticket counter) runs the one inverse real FFT and writes FCS_d.
//
// Three engines:
//   cp_run<L, NT, CPT>           P = 2^(L+1) <= 8192 on the slot FFT of
//                                fcs_fft.cuh (NT = 2^(L-4) threads, 16 points
//                                each, >= 32);
//   cp12_run<CPT, RMAX>          P = 8192 on the warp-DIT engine of
//                                fcs_dit.cuh (256 threads, two block barriers
//                                per transform);
//   cp_pair_run<NR, CPT>         P = 1024 NR = 16384 or 32768 on the row-pair
//                                engine of fcs_pair.cuh (two block barriers
//                                per transform).
//
// The problem is read through a small accessor interface (Prob):
//   int modes(), int64_t dim(n), const float *column(n, r), float
//   value(column, i, n, r) (its entry i), int range(n) (J_n) and void ready()
//   (called before the first access to any of these) (value and ready for
//   cp_pair_run only, range for it and cp12_run),
//   const int32_t *hashes(d, n), const int8_t *signs(d, n), int64_t length(),
//   float *sketch(d), float2 *spectrum() ([D][M + 2] float2, 16-byte
//   aligned, zero before the first group of a sketch adds into it),
//   unsigned *ticket(d) (zero at start; reset by the last group), int sb
//   (scatter-buffer length in floats: max J_n rounded up to 4).
#pragma once

#include <type_traits>

#include "fcs_dit.cuh"
#include "fcs_pair.cuh"

namespace fcs {

// Shared-memory layout of cp_run; every region starts on a 16-byte
// boundary (the scatter buffer is cleared with float4 stores).
template <int LOG2M, int NT>
struct CpSmem {
  static constexpr size_t up16(size_t x) { return (x + 15) & ~size_t(15); }
  static constexpr size_t kB = 0;
  static constexpr size_t kAcc = up16(kB + sizeof(float2) * padded_len(1 << LOG2M));
  static constexpr size_t kTw =
      up16(kAcc + sizeof(float2) * LastPass<LOG2M, NT>::NV * NT);
  static constexpr size_t kA = up16(kTw + sizeof(float2) * plan_twlen(LOG2M));
  static size_t bytes(int sb) { return kA + sizeof(float) * size_t(sb); }
};

// Ranks [r0, r1) of sketch d on the slot FFT (M = 2^LOG2M complex points,
// NT threads).  CPT = factor entries prefetched per thread (the rest of a
// longer column is scattered by a direct loop); `groups` = number of groups
// that add into sketch d.  Every thread of the block calls it; it returns
// with no barrier pending.
template <int LOG2M, int NT, int CPT, class Prob>
__device__ __forceinline__ void cp_run(const Prob &a, int d, int64_t r0, int64_t r1,
                                       unsigned groups, unsigned char *smem_raw,
                                       const float2 *__restrict__ tw, int *is_last) {
  using LPs = LastPass<LOG2M, NT>;
  constexpr int M = 1 << LOG2M;
  constexpr int HALF = M / 2;
  constexpr int RL = LPs::RL, EPS = LPs::EPS, NV = LPs::NV;
  using Lay = CpSmem<LOG2M, NT>;
  float2 *B = reinterpret_cast<float2 *>(smem_raw + Lay::kB);      // padded_len(M)
  float2 *accS = reinterpret_cast<float2 *>(smem_raw + Lay::kAcc); // NV * NT
  float2 *tws = reinterpret_cast<float2 *>(smem_raw + Lay::kTw);   // plan_twlen
  float *A = reinterpret_cast<float *>(smem_raw + Lay::kA);        // sb floats
  const int tid = threadIdx.x;
  const int N = a.modes();
  const int sb = a.sb;

  fill_twiddles<LOG2M, NT>(tws, tw);
  LastPassTw<LOG2M, NT> ltw;
  ltw.load(tw);
  for (int e = tid; e < sb / 4; e += NT) reinterpret_cast<float4 *>(A)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int v = 0; v < NV; ++v) accS[v * NT + tid] = make_float2(0.f, 0.f);

  // prefetched column: signed factor values and hash bins
  float pv[CPT];
  int ph[CPT];
  auto fetch = [&](int64_t r, int n) {
    const int64_t In = a.dim(n);
    const float *col = a.column(n, r);
    const int32_t *hn = a.hashes(d, n);
    const int8_t *sn = a.signs(d, n);
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
      const int64_t i = tid + int64_t(c) * NT;
      ph[c] = -1;
      pv[c] = 0.f;
      if (i < In) {
        const float v = a.ld(col + i);
        pv[c] = a.ld(sn + i) < 0 ? -v : v;
        ph[c] = a.ld(hn + i);
      }
    }
  };
  fetch(r0, 0);
  __syncthreads();

  float2 X[EPS][2][RL], p[EPS][2][RL];
  for (int64_t r = r0; r < r1; ++r) {
    for (int n = 0; n < N; ++n) {
#pragma unroll
      for (int c = 0; c < CPT; ++c)
        if (unsigned(ph[c]) < unsigned(sb)) atomicAdd(A + ph[c], pv[c]);
      const int64_t In = a.dim(n);
      if (In > int64_t(CPT) * NT) {
        // entries beyond the prefetched chunk: load and scatter directly
        const float *col = a.column(n, r);
        const int32_t *hn = a.hashes(d, n);
        const int8_t *sn = a.signs(d, n);
        for (int64_t i = int64_t(CPT) * NT + tid; i < In; i += NT) {
          const int hb = a.ld(hn + i);
          const float v = a.ld(col + i);
          if (unsigned(hb) < unsigned(sb)) atomicAdd(A + hb, a.ld(sn + i) < 0 ? -v : v);
        }
      }
      // prefetch the next column while this one is transformed
      if (n + 1 < N)
        fetch(r, n + 1);
      else if (r + 1 < r1)
        fetch(r + 1, 0);
      __syncthreads();
      fft_first_pass<LOG2M, NT>(A, sb, B);
      __syncthreads();
      for (int e = tid; e < sb / 4; e += NT)
        reinterpret_cast<float4 *>(A)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      fft_middle_passes<LOG2M, NT, 1>(B, tws);
      fft_last_pass_unpack<LOG2M, NT>(B, ltw, X);
#pragma unroll
      for (int e = 0; e < EPS; ++e)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int q = 0; q < RL; ++q) {
            if (n == 0) {
              p[e][b][q] = X[e][b][q];
            } else {
              const bool packed = (b == 0 && q == 0 && tid + e * NT == 0);
              p[e][b][q] = slot_mul(p[e][b][q], X[e][b][q], packed);
            }
          }
    }
#pragma unroll
    for (int e = 0; e < EPS; ++e)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int q = 0; q < RL; ++q) {
          float2 &acc = accS[((e * 2 + b) * RL + q) * NT + tid];
          acc = cadd(acc, p[e][b][q]);
        }
  }

  // publish the partial spectrum
  float2 *Gd = a.spectrum() + d * int64_t(M + 2);
#pragma unroll
  for (int e = 0; e < EPS; ++e) {
    if (LPs::SLOTS % NT != 0 && tid + e * NT >= LPs::SLOTS) continue;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int q = 0; q < RL; ++q) {
        const float2 v = accS[((e * 2 + b) * RL + q) * NT + tid];
        const int k = last_pass_index<LOG2M, NT>(e, b, q);
        if (k == 0) {
          atomicAdd(&Gd[0].x, v.x);
          atomicAdd(&Gd[M].x, v.y);
        } else {
          atomicAdd(&Gd[k], v);
        }
      }
  }
  __threadfence();
  __syncthreads();
  unsigned *ticket = a.ticket(d);
  if (tid == 0) *is_last = (atomicAdd(ticket, 1u) == groups - 1);
  __syncthreads();
  if (!*is_last) return;
  __threadfence();

  // last group for sketch d: one inverse real FFT of the summed spectrum
  for (int q = tid; q < HALF; q += NT) {
    float2 Av, Bv;
    if (q == 0) {
      Av = make_float2(__ldcg(&Gd[0].x), __ldcg(&Gd[M].x));
      Bv = __ldcg(&Gd[HALF]);
    } else {
      Av = __ldcg(&Gd[q]);
      Bv = __ldcg(&Gd[M - q]);
    }
    pack_pair_conj<LOG2M>(B, q, Av, Bv, tw);
  }
  __syncthreads();
  block_fft<LOG2M, NT>(B, tw);
  const float sc = 1.0f / float(M);
  float *od = a.sketch(d);
  const int64_t Jt = a.length();
  float *Br = reinterpret_cast<float *>(B);
  for (int64_t j = tid; j < Jt; j += NT) {
    const float v = Br[real_off(int(j))];
    od[j] = (j & 1) ? -v * sc : v * sc;
  }
  if (tid == 0) *ticket = 0u;
}

// Shared-memory layout of cp12_run; ra = number of float2 columns of the
// 8-row scatter buffer.
struct Cp12Smem {
  static constexpr size_t kB = 0;                                   // 8 x kRS float2
  static constexpr size_t kTw = kB + sizeof(float2) * 8 * wdit::kRS;
  static constexpr size_t kA = kTw + sizeof(float2) * wdit::kTwLen;
  static size_t bytes(int ra) { return kA + sizeof(float2) * 8 * size_t(ra); }
};

// Ranks [r0, r1) of sketch d for P = 8192 on the warp-DIT engine of
// fcs_dit.cuh (256 threads): per transform the Count Sketch goes into an 8-row
// scatter buffer, warp w runs the 512-point FFT of row w, one block barrier,
// then each thread transforms its two columns and unpacks them in registers
// (TWICE the spectrum values, so the inverse scales by 2^-N).  The mode
// product and the rank sum stay in registers; the next column is scattered
// between the barriers by half the warps before step 2 and half after.  CPT
// and `groups` as for cp_run; RMAX = number of 32-entry blocks per
// scatter-buffer row (ra <= 32 RMAX).  Every thread of the 256-thread block
// calls it; it returns with no barrier pending.
template <int CPT, int RMAX, class Prob>
__device__ __forceinline__ void cp12_run(const Prob &a, int d, int64_t r0, int64_t r1,
                                         unsigned groups, unsigned char *smem_raw,
                                         const float2 *__restrict__ tw, int *is_last) {
  namespace W = wdit;
  constexpr int NT = W::kNT, M = W::kM, HALF = M / 2;
  float2 *B = reinterpret_cast<float2 *>(smem_raw + Cp12Smem::kB);
  float2 *tws = reinterpret_cast<float2 *>(smem_raw + Cp12Smem::kTw);
  float2 *A2 = reinterpret_cast<float2 *>(smem_raw + Cp12Smem::kA);
  float *A = reinterpret_cast<float *>(A2);
  const int tid = threadIdx.x, warp = tid >> 5;
  const int N = a.modes();
  const int sb = a.sb;
  const int ra = (sb + 15) >> 4;
  const int ua = W::ua_of(tid), ub = W::ub_of(tid);

  float pv[CPT];
  int ph[CPT];
  auto fetch = [&](int64_t r, int n) {
    const int64_t In = a.dim(n);
    const float *col = a.column(n, r);
    const int32_t *hn = a.hashes(d, n);
    const int8_t *sn = a.signs(d, n);
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
      const int64_t i = tid + int64_t(c) * NT;
      ph[c] = -1;
      pv[c] = 0.f;
      if (i < In) {
        const float v = a.ld(col + i);
        pv[c] = a.ld(sn + i) < 0 ? -v : v;
        ph[c] = a.ld(hn + i);
      }
    }
  };
  auto scatter = [&](int64_t r, int n) {
#pragma unroll
    for (int c = 0; c < CPT; ++c)
      if (unsigned(ph[c]) < unsigned(a.range(n))) atomicAdd(A + W::a_index(ph[c], ra), pv[c]);
    const int64_t In = a.dim(n);
    if (In > int64_t(CPT) * NT) {
      const float *col = a.column(n, r);
      const int32_t *hn = a.hashes(d, n);
      const int8_t *sn = a.signs(d, n);
      for (int64_t i = int64_t(CPT) * NT + tid; i < In; i += NT) {
        const int hb = a.ld(hn + i);
        const float v = a.ld(col + i);
        if (unsigned(hb) < unsigned(a.range(n)))
          atomicAdd(A + W::a_index(hb, ra), a.ld(sn + i) < 0 ? -v : v);
      }
    }
  };
  fetch(r0, 0);
  W::fill_twiddles(tws, tw);
  for (int e = tid; e < 8 * ra; e += NT) A2[e] = make_float2(0.f, 0.f);
  __syncthreads();
  scatter(r0, 0);
  __syncthreads();

  float2 pa[8], pb[8], acca[8], accb[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acca[j] = accb[j] = make_float2(0.f, 0.f);
  for (int64_t r = r0; r < r1; ++r) {
    for (int n = 0; n < N; ++n) {
      int64_t rn = r;
      int nn = n + 1;
      if (nn == N) {
        nn = 0;
        ++rn;
      }
      const bool more = rn < r1;
      if (more) fetch(rn, nn);
      wdit::step1_row<RMAX, false, false>(A2 + warp * ra, ra, B + warp * wdit::kRS, tws, warp);
      __syncthreads();
      const bool early = tid < NT / 2;
      if (more && early) scatter(rn, nn);
      float2 va[8], vb[8];
      W::step2(B, tws, va, vb);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (n == 0) {
          pa[j] = va[j];
          pb[j] = vb[j];
        } else {
          pa[j] = cmul(pa[j], va[j]);
          pb[j] = slot_mul(pb[j], vb[j], tid == 0 && j == 0);
        }
      }
      if (n == N - 1) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          acca[j] = cadd(acca[j], pa[j]);
          accb[j] = cadd(accb[j], pb[j]);
        }
      }
      if (more && !early) scatter(rn, nn);
      __syncthreads();
    }
  }

  // publish the partial spectrum: bins ua + 512 j and ub + 512 j (thread 0:
  // ub = 0, whose j = 0 value packs the real bins 0 and M)
  float2 *Gd = a.spectrum() + d * int64_t(M + 2);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    atomicAdd(&Gd[ua + 512 * j], acca[j]);
    if (tid == 0 && j == 0) {
      atomicAdd(&Gd[0].x, accb[0].x);
      atomicAdd(&Gd[M].x, accb[0].y);
    } else {
      atomicAdd(&Gd[ub + 512 * j], accb[j]);
    }
  }
  __threadfence();
  __syncthreads();
  unsigned *ticket = a.ticket(d);
  if (tid == 0) *is_last = (atomicAdd(ticket, 1u) == groups - 1);
  __syncthreads();
  if (!*is_last) return;
  __threadfence();

  // last group for sketch d: the conj-packed sequence of the summed spectrum,
  // row-swizzled into B, a forward complex FFT in place, conj and scaling
  {
    constexpr int PER = HALF / NT;
    float2 Av[PER], Bv[PER], Wv[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int q = k * NT + tid;
      if (q == 0) {
        Av[k] = make_float2(__ldcg(&Gd[0].x), __ldcg(&Gd[M].x));
        Bv[k] = __ldcg(&Gd[HALF]);
        Wv[k] = make_float2(1.f, 0.f);
      } else {
        Av[k] = __ldcg(&Gd[q]);
        Bv[k] = __ldcg(&Gd[M - q]);
        Wv[k] = __ldg(&tw[q << (kLogTwN - 13)]);      // W_P^q, P = 8192
      }
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int q = k * NT + tid;
      float2 cq, cm;
      pack_pair_conj_values_w(q, Av[k], Bv[k], Wv[k], cq, cm);
      B[W::row_pos_swz(q)] = cq;
      B[W::row_pos_swz(q ? M - q : HALF)] = cm;
    }
  }
  __syncthreads();
  wdit::step1_row<16, true, true>(B + warp * wdit::kRS, 512, B + warp * wdit::kRS, tws, warp);
  __syncthreads();
  float2 va[8], vb[8];
  W::step2_complex(B, tws, va, vb);                  // Z[ua + 512 q1], Z[ub + 512 q1]
  // 1/M of the inverse and 2^-N for the doubled unpack of every mode
  const float sc = 1.0f / (float(M) * float(1 << N));
  float *od = a.sketch(d);
  const int64_t Jt = a.length();
#pragma unroll
  for (int q1 = 0; q1 < 8; ++q1) {
    const int64_t ma = ua + 512 * q1, mb = ub + 512 * q1;
    if (2 * ma < Jt) od[2 * ma] = va[q1].x * sc;
    if (2 * ma + 1 < Jt) od[2 * ma + 1] = -va[q1].y * sc;
    if (2 * mb < Jt) od[2 * mb] = vb[q1].x * sc;
    if (2 * mb + 1 < Jt) od[2 * mb + 1] = -vb[q1].y * sc;
  }
  if (tid == 0) *ticket = 0u;
}

// The ranks one block takes, one after another: first() (known at once), then
// those request() asks for -- one thread, one rank ahead -- and get() reads
// after a block barrier; done(r) past the end.
struct RankRange {                       // [r0, r1)
  int64_t r0, r1;
  __device__ __forceinline__ int64_t first() const { return r0; }
  __device__ __forceinline__ int64_t second() const { return r0 + 1; }
  __device__ __forceinline__ void request(int64_t) const {}
  __device__ __forceinline__ int64_t get(int64_t next) const { return next + 1; }
  __device__ __forceinline__ bool done(int64_t r) const { return r >= r1; }
};
// From a counter shared by the `groups` blocks of a sketch (zero at the
// start), so that a block whose SM is less busy takes more of them.
struct RankQueue {
  int64_t R;
  unsigned groups, g;
  unsigned long long *counter;           // global
  int64_t *slot;                         // shared
  __device__ __forceinline__ int64_t first() const { return g; }
  __device__ __forceinline__ int64_t second() const {     // every thread; ends with a barrier
    request(0);
    __syncthreads();
    return *slot;
  }
  __device__ __forceinline__ void request(int64_t) const {
    if (threadIdx.x == 0) *slot = int64_t(groups + atomicAdd(counter, 1ull));
  }
  __device__ __forceinline__ int64_t get(int64_t) const { return *slot; }
  __device__ __forceinline__ bool done(int64_t r) const { return r >= R; }
};

// The given ranks of sketch d for P = 1024 NR on the row-pair engine of
// fcs_pair.cuh: per transform the Count Sketch goes into the row-pair scatter
// buffer, each warp transforms its row pairs, one block barrier, then each
// thread transforms and unpacks its two columns (TWICE the spectrum values,
// so the inverse scales by 2^-N).  The mode product and the rank sum are in
// tensor memory (`tm`: this CTA's allocation).  The next column is scattered
// between the barriers by half the warps before the column step and half
// after.  CPT and `groups` as for cp_run.  Every thread of the block calls it;
// it returns with no barrier pending.
//
// Bound: the FP32 pipe and the shared-memory pipe, together with the waits
// between them: at P = 16384 a transform takes 5.4 k clocks of an SM, of which
// each pipe needs 3.4 k (1900 packed FP32 instructions per scheduler, 3400
// shared wavefronts).  Over a whole launch (I = 1000, R = 100, D = 10) the FMA pipe is
// 43 % busy, the shared pipe 53 %, issue 45 %.
template <int NR, int CPT, class Prob, class Ranks>
__device__ __forceinline__ void cp_pair_run(const Prob &a, int d, const Ranks &ranks,
                                            unsigned groups, unsigned char *smem_raw,
                                            const float2 *__restrict__ tw, int *is_last,
                                            uint32_t tm) {
  using Geo = pfft::Geo<NR>;
  using Lay = pfft::Smem<NR>;
  constexpr int NT = Geo::NT, M = Geo::M, HALF = M / 2, H = Geo::H;
  float4 *B = reinterpret_cast<float4 *>(smem_raw + Lay::kB);
  float2 *t0 = reinterpret_cast<float2 *>(smem_raw + Lay::kT0);
  float2 *t1 = reinterpret_cast<float2 *>(smem_raw + Lay::kT1);
  float2 *t2 = reinterpret_cast<float2 *>(smem_raw + Lay::kT2);
  float2 *t3 = reinterpret_cast<float2 *>(smem_raw + Lay::kT3);
  float4 *A4 = reinterpret_cast<float4 *>(smem_raw + Lay::kA);
  float *A = reinterpret_cast<float *>(A4);
  const int tid = threadIdx.x, warp = tid >> 5;
  const int N = a.modes();
  const int sb = a.sb;
  const int ra = (sb + 2 * NR - 1) / (2 * NR);

  float pv[CPT];
  int ph[CPT];
  auto fetch = [&](int64_t r, int n) {
    const int64_t In = a.dim(n);
    const float *col = a.column(n, r);
    const int32_t *hn = a.hashes(d, n);
    const int8_t *sn = a.signs(d, n);
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
      const int64_t i = tid + int64_t(c) * NT;
      ph[c] = -1;
      pv[c] = 0.f;
      if (i < In) {
        const float v = a.value(col, i, n, r);
        pv[c] = a.ld(sn + i) < 0 ? -v : v;
        ph[c] = a.ld(hn + i);
      }
    }
  };
  auto scatter = [&](int64_t r, int n) {
#pragma unroll
    for (int c = 0; c < CPT; ++c)
      if (unsigned(ph[c]) < unsigned(a.range(n)))
        atomicAdd(A + pfft::a_index<NR>(ph[c], ra), pv[c]);
    const int64_t In = a.dim(n);
    if (In > int64_t(CPT) * NT) {
      const float *col = a.column(n, r);
      const int32_t *hn = a.hashes(d, n);
      const int8_t *sn = a.signs(d, n);
#pragma unroll 4
      for (int64_t i = int64_t(CPT) * NT + tid; i < In; i += NT) {
        const int hb = a.ld(hn + i);
        const float v = a.value(col, i, n, r);
        if (unsigned(hb) < unsigned(a.range(n)))
          atomicAdd(A + pfft::a_index<NR>(hb, ra), a.ld(sn + i) < 0 ? -v : v);
      }
    }
  };
  pfft::fill_twiddles<NR>(smem_raw, tw);
  for (int e = tid; e < H * ra; e += NT) A4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  a.ready();
  int64_t r = ranks.first();
  fetch(r, 0);
  int64_t rnext = ranks.second();
  __syncthreads();
  scatter(r, 0);
  __syncthreads();

  const uint32_t tp = pfft::tmem_mine<NR>(tm), ts = tp + Geo::WPT;   // product, rank sum
  const bool w0 = warp == Geo::WARPS - 1;            // the warp that has column 0
  float2 p0 = make_float2(0.f, 0.f), s0 = p0;
  // column pair c of the current transform: product and rank sum.  The
  // tensor-memory loads of a group of values are issued a group ahead.
  auto columns = [&](int c, bool product, bool last, bool sum) {
    pfft::C2 xa[H], xc[H];
    pfft::column_step<NR>(B, t2, c, xa, xc);
    const uint32_t op = tp + uint32_t(c) * (8 * H), os = ts + uint32_t(c) * (8 * H);
    __syncwarp();                                    // tensor-memory accesses are warp-wide
    pfft::Tm16 x;
    if (product) pfft::tmem_ld16(op, x);
    pfft::unpack<NR>(t2, c, xa, xc);
#pragma unroll
    for (int g = 0; g < 2 * H; g += 4) {             // four value pairs: 16 words
      pfft::C2 v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = g < H ? xa[g + i] : xc[g - H + i];
      if (product) {
        pfft::tmem_wait_ld(x);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = pfft::cmul(pfft::tm_get(x, i), v[i]);
      }
      pfft::Tm16 y;
      if (sum) pfft::tmem_ld16(os + 4 * g, y);
      if (product && g + 4 < 2 * H) pfft::tmem_ld16(op + 4 * (g + 4), x);
      if (sum) {
        pfft::tmem_wait_ld(y);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = pfft::cadd(v[i], pfft::tm_get(y, i));
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) pfft::tm_set(y, i, v[i]);
      pfft::tmem_st16((last ? os : op) + 4 * g, y);
    }
  };
  for (bool first_rank = true;; first_rank = false) {
    int64_t rnext2 = rnext;
    for (int n = 0; n < N; ++n) {
      const bool wrap = n + 1 == N;
      const int nn = wrap ? 0 : n + 1;
      const int64_t rn = wrap ? rnext : r;
      const bool more = !ranks.done(rn);
      if (n == 0) ranks.request(rnext);
      if (more) fetch(rn, nn);
      pfft::scatter_row_step<Geo::RPW, Geo::PAD>(A4 + warp * ra, Geo::WARPS * ra, ra,
                                                 B + warp * Geo::RS, Geo::WARPS * Geo::RS, t0, t1);
      __syncthreads();
      if (n == 0) rnext2 = ranks.get(rnext);
      const bool early = tid < NT / 2;
      if (more && early) scatter(rn, nn);
      if (w0) {
        const float2 x = pfft::column0<NR>(B, t3);
        p0 = n == 0 ? x : slot_mul(p0, x, (tid & 31) == 0);
        if (wrap) s0 = cadd(s0, p0);
      }
#pragma unroll 1
      for (int c = 0; c < Geo::NCP; ++c) columns(c, n > 0, wrap, wrap && !first_rank);
      pfft::tmem_wait_st();
      if (more && !early) scatter(rn, nn);
      __syncthreads();
    }
    r = rnext;
    rnext = rnext2;
    if (ranks.done(r)) break;
  }

  // publish the partial spectrum (2^N X in natural order) through B, as
  // 16-byte atomics
  float2 *Gd = a.spectrum() + d * int64_t(M + 2);
  float2 *Bs = reinterpret_cast<float2 *>(B);
#pragma unroll 1
  for (int c = 0; c < Geo::NCP; ++c) {
#pragma unroll
    for (int g = 0; g < 2 * H; g += 4) {
      pfft::Tm16 x;
      pfft::tmem_ld16(ts + uint32_t(c) * (8 * H) + 4 * g, x);
      pfft::tmem_wait_ld(x);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        // (u = 256 writes its bins twice, the same value up to rounding)
        const pfft::C2 v = pfft::tm_get(x, i);
        const int b = g < H ? 0 : 1, k = g < H ? g + i : (2 * H - (g + i)) % H;
        Bs[pfft::bin_of<NR>(c, b, k, 0)] = make_float2(pfft::lo(v.re), pfft::lo(v.im));
        Bs[pfft::bin_of<NR>(c, b, k, 1)] = make_float2(pfft::hi(v.re), pfft::hi(v.im));
      }
    }
  }
  if (w0 && (tid & 31) < NR) {
    const int i = tid & 31;
    Bs[512 * i] = make_float2(s0.x, i ? s0.y : 0.f);
    if (i == 0) Bs[M] = make_float2(s0.y, 0.f);
  }
  __syncthreads();
  // the blocks of a sketch end together: each starts at another of 32 places,
  // or they queue up at the same lines (6.3 us a block instead of 2.6 at P = 16384, D = 10)
  const int f0 = ((blockIdx.x * 37) & 31) * (M / 64) + tid;
  for (int f = 0; f < M / 2; f += NT) {
    const int e = (f0 + f) & (M / 2 - 1);
    atomicAdd(reinterpret_cast<float4 *>(Gd) + e, B[e]);
  }
  if (tid == 0) atomicAdd(&Gd[M].x, Bs[M].x);
  __threadfence();
  __syncthreads();
  unsigned *ticket = a.ticket(d);
  if (tid == 0) *is_last = (atomicAdd(ticket, 1u) == groups - 1);
  __syncthreads();
  if (!*is_last) return;
  __threadfence();

  // last group for sketch d: the conj-packed sequence of the summed spectrum
  // into B, a forward complex FFT in place, conj and scaling
  float *Bf = reinterpret_cast<float *>(B);
  auto put = [&](int m, float2 z) {
    float *p = Bf + pfft::b_index<NR>(m);
    p[0] = z.x;
    p[2] = z.y;
  };
  constexpr int BATCH = NR == 32 ? 16 : 8;
  for (int q0 = tid; q0 < HALF; q0 += BATCH * NT) {
    float2 Av[BATCH], Bv[BATCH], Wv[BATCH];
#pragma unroll
    for (int k = 0; k < BATCH; ++k) {
      const int q = q0 + k * NT;
      if (q == 0) {
        Av[k] = make_float2(__ldcg(&Gd[0].x), __ldcg(&Gd[M].x));
        Bv[k] = __ldcg(&Gd[HALF]);
        Wv[k] = make_float2(1.f, 0.f);
      } else {
        Av[k] = __ldcg(&Gd[q]);
        Bv[k] = __ldcg(&Gd[M - q]);
        Wv[k] = __ldg(&tw[q << (kLogTwN - Geo::LM - 1)]);   // W_P^q
      }
    }
#pragma unroll
    for (int k = 0; k < BATCH; ++k) {
      const int q = q0 + k * NT;
      float2 cq, cm;
      pack_pair_conj_values_w(q, Av[k], Bv[k], Wv[k], cq, cm);
      put(q, cq);
      put(q ? M - q : HALF, cm);
    }
  }
  __syncthreads();
  pfft::row_step<32, true, Geo::RPW, Geo::PAD>(B + warp * Geo::RS, Geo::WARPS * Geo::RS, 512,
                                               B + warp * Geo::RS, Geo::WARPS * Geo::RS, t0, t1);
  __syncthreads();
  // 1/M of the inverse and 2^-N for the doubled unpack of every mode
  const float sc = 1.0f / (float(M) * float(1 << N));
  float *od = a.sketch(d);
  const int64_t Jt = a.length();
  auto emit = [&](int m, float x, float y) {
    if (2 * m < Jt) od[2 * m] = x * sc;
    if (2 * m + 1 < Jt) od[2 * m + 1] = -y * sc;
  };
#pragma unroll 1
  for (int c = 0; c < Geo::NCP; ++c) {
    const int u = tid + 1 + c * NT, uc = 512 - u;
    pfft::C2 xa[H], xc[H];
    pfft::column_step<NR>(B, t2, c, xa, xc);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      emit(u + 512 * k, pfft::lo(xa[k].re), pfft::lo(xa[k].im));
      emit(u + 512 * (k + H), pfft::hi(xa[k].re), pfft::hi(xa[k].im));
      // C[q1 + 1] is the second column's element q1
      const int ql = (k == 0 ? NR - 1 : k + H - 1), qh = (k == 0 ? H - 1 : k - 1);
      emit(uc + 512 * ql, pfft::lo(xc[k].re), pfft::lo(xc[k].im));
      emit(uc + 512 * qh, pfft::hi(xc[k].re), pfft::hi(xc[k].im));
    }
  }
  if (w0 && (tid & 31) < NR) {
    const float2 z = pfft::column0_complex<NR>(B, t3);
    emit(512 * (tid & 31), z.x, z.y);
  }
  if (tid == 0) *ticket = 0u;
}

}  // namespace fcs
