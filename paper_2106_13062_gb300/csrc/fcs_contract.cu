// fcs_contract.cu -- fcs_contract: the sketched contractions of Sec. 4.1.
//
//  ALL  (eq. T_uvw):  e_d = <FCS_d(T), FCS_d(v_1 o ... o v_N)>
//       = (1/P) Re sum_{k<P} conj(F(FCS_d T))[k] prod_n F(CS_n v_n)[k]
//       (Parseval; FCS_d of the rank-1 tensor is the product of the per-mode
//       spectra by eq. FCS_syn with R = 1).
//  FREE (eq. T_Ivw, free mode m; also the ALS columns of Sec. 4.1.2):
//       z_d = IFFT(F(FCS_d T) prod_{n != m} conj F(CS_n v_n)),
//       est_d[i] = s_m(i) z_d[h_m(i)]   (exact for P >= Jt: the circular
//       correlation never wraps at the lags h_m(i) < J_m).
//  Then the median over the D sketches (Sec. 4 opening).
//
// Kernels: (1) the half spectra of the D sketches of T; (2) one CTA per
// (batch item, sketch) that builds each needed Count Sketch in shared memory,
// transforms it and folds it into the per-thread spectrum product, then either
// reduces the Parseval sum or runs the inverse FFT and gathers; (3) the median
// (of both results in one launch).  (2) runs on the slot FFT of fcs_fft.cuh
// and, for large batches at P = 16384, on the row-pair engine of fcs_pair.cuh.
// Each kernel is launched so that it may start before the one before has
// ended and waits where it first reads what that one wrote.
//
// With fcs_cache_spectra enabled, the spectra of (1) are kept in a
// per-context cache keyed by the sketch pointer and shape, so repeated
// contractions against one sketch (the RTPM and ALS loops) transform it
// once.  fcs_forget drops an entry; the library's own sketch calls drop the
// entries of the buffers they overwrite.
#include <vector>

#include "fcs_pair.cuh"

struct fcs_spec_cache {
  struct Entry {
    const float *key;
    int64_t Jt;
    int D;
    int log2m;
    float2 *spec;
    size_t bytes;
    cudaEvent_t ready;   // spectrum written
    cudaEvent_t used;    // last contraction that read it
    uint64_t tick;
    bool stale;          // key's contents may have changed: recompute on next use
  };
  std::vector<Entry> e;
  size_t bytes = 0;
  uint64_t tick = 0;
};

namespace fcs {
namespace {

constexpr int kSpecCacheEntries = 16;
constexpr size_t kSpecCacheMaxBytes = size_t(512) << 20;

void spec_entry_free(fcs_spec_cache::Entry &x) {
  cudaEventSynchronize(x.used);
  cudaEventDestroy(x.ready);
  cudaEventDestroy(x.used);
  cudaFree(x.spec);
}

void spec_cache_erase(fcs_spec_cache *c, size_t i) {
  spec_entry_free(c->e[i]);
  c->bytes -= c->e[i].bytes;
  c->e.erase(c->e.begin() + i);
}

// Entry for (key, Jt, D, log2m): an existing one (hit = true) or a new one
// whose spectrum the caller must compute; nullptr when it cannot be cached.
fcs_spec_cache::Entry *spec_cache_get(fcs_ctx *ctx, const float *key, int64_t Jt, int D,
                                      int log2m, bool *hit) {
  *hit = false;
  if (!ctx->cache_spectra) return nullptr;
  if (!ctx->spec_cache) ctx->spec_cache = new (std::nothrow) fcs_spec_cache();
  fcs_spec_cache *c = ctx->spec_cache;
  if (!c) return nullptr;
  ++c->tick;
  for (auto &x : c->e) {
    if (x.key == key && x.Jt == Jt && x.D == D && x.log2m == log2m) {
      x.tick = c->tick;
      if (x.stale) {
        // recompute into the same memory once its last readers are done
        if (cudaStreamWaitEvent(ctx->stream, x.used, 0) != cudaSuccess) {
          cudaGetLastError();
          return nullptr;
        }
        x.stale = false;
        return &x;
      }
      *hit = true;
      return &x;
    }
  }
  const size_t bytes = sizeof(float2) * size_t(D) * ((size_t(1) << log2m) + 1);
  const size_t cap = ctx->budget / 2 < kSpecCacheMaxBytes ? ctx->budget / 2 : kSpecCacheMaxBytes;
  if (bytes > cap) return nullptr;
  while (!c->e.empty() && (c->bytes + bytes > cap || int(c->e.size()) >= kSpecCacheEntries)) {
    size_t lru = 0;
    for (size_t i = 1; i < c->e.size(); ++i)
      if (c->e[i].tick < c->e[lru].tick) lru = i;
    spec_cache_erase(c, lru);
  }
  fcs_spec_cache::Entry x{key, Jt, D, log2m, nullptr, bytes, nullptr, nullptr, c->tick, false};
  if (cudaMalloc(&x.spec, bytes) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  if (cudaEventCreateWithFlags(&x.ready, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&x.used, cudaEventDisableTiming) != cudaSuccess) {
    cudaGetLastError();
    if (x.ready) cudaEventDestroy(x.ready);
    cudaFree(x.spec);
    return nullptr;
  }
  c->e.push_back(x);
  c->bytes += bytes;
  return &c->e.back();
}

struct ContractArgs {
  Modes m;
  int D;
  int kind;
  int free_mode;
  int64_t B;
  const float *fcsT;      // [D][Jt]
  const float *vec[kMaxN];
  const int32_t *h;
  const int8_t *s;
  float2 *spec;           // [D][M+1]
  float *raw;             // [B][D] or [B][D][I_m]
  float *raw_all;         // kBoth: the T(v_1..v_N) estimates [B][D]
  float *out;             // [B] or [B][I_m]
  int sb;                 // compact count-sketch buffer (floats, multiple of 4)
};

// Half spectrum of each of the D sketches of T, natural order [D][M+1]: the
// sketch is read into the compact real buffer and transformed by the block
// real FFT whose last pass leaves the spectrum in registers.
template <int LOG2M, int NT>
__global__ void __launch_bounds__(NT) spectrum_kernel(const float *__restrict__ x, int64_t len,
                                                      int64_t ld, int sb,
                                                      float2 *__restrict__ spec,
                                                      const float2 *__restrict__ tw) {
  using LPs = LastPass<LOG2M, NT>;
  using Lay = FftSmem<LOG2M>;
  constexpr int M = 1 << LOG2M;
  constexpr int RL = LPs::RL, EPS = LPs::EPS;
  extern __shared__ __align__(16) unsigned char smem[];
  float2 *B = reinterpret_cast<float2 *>(smem + Lay::kB);
  float2 *tws = reinterpret_cast<float2 *>(smem + Lay::kTw);
  float *A = reinterpret_cast<float *>(smem + Lay::kA);
  const float *xd = x + blockIdx.x * ld;
  griddep_launch();
  fill_twiddles<LOG2M, NT>(tws, tw);
  float2 *lps = reinterpret_cast<float2 *>(smem + Lay::kLp);
  LastPassTwShared<LOG2M, NT>::fill(lps, tw);
  const LastPassTwShared<LOG2M, NT> ltw{lps};
  for (int j = threadIdx.x; j < sb; j += NT) A[j] = j < len ? __ldg(xd + j) : 0.f;
  float2 X[EPS][2][RL];
  rfft_to_slots<LOG2M, NT>(A, sb, B, tws, ltw, X);
  float2 *sd = spec + blockIdx.x * int64_t(M + 1);
#pragma unroll
  for (int e = 0; e < EPS; ++e) {
    if (LPs::SLOTS % NT != 0 && int(threadIdx.x) + e * NT >= LPs::SLOTS) continue;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        const int q = last_pass_index<LOG2M, NT>(e, b, r);
        if (q == 0) {
          sd[0] = make_float2(X[e][b][r].x, 0.f);
          sd[M] = make_float2(X[e][b][r].y, 0.f);
        } else {
          sd[q] = X[e][b][r];
        }
      }
  }
}

// Internal kind: both contractions of one vector set from one set of
// transforms (fcs_contract_both).
constexpr int kBoth = 2;

template <int LOG2M, int NT>
__global__ void __launch_bounds__(NT) contract_kernel(ContractArgs a,
                                                      const float2 *__restrict__ tw) {
  using LPs = LastPass<LOG2M, NT>;
  using Lay = FftSmem<LOG2M>;
  constexpr int M = 1 << LOG2M;
  constexpr int RL = LPs::RL, EPS = LPs::EPS;
  extern __shared__ __align__(16) unsigned char smem[];
  float2 *B = reinterpret_cast<float2 *>(smem + Lay::kB);
  float2 *tws = reinterpret_cast<float2 *>(smem + Lay::kTw);
  float *A = reinterpret_cast<float *>(smem + Lay::kA);
  __shared__ float red[NT / 32];
  const int tid = threadIdx.x;
  const int64_t b = blockIdx.x;
  const int d = blockIdx.y;
  const bool all = a.kind == FCS_CONTRACT_ALL;
  const int sb = a.sb;
  const float2 *sd = a.spec + d * int64_t(M + 1);
  fill_twiddles<LOG2M, NT>(tws, tw);
  float2 *lps = reinterpret_cast<float2 *>(smem + Lay::kLp);
  LastPassTwShared<LOG2M, NT>::fill(lps, tw);
  const LastPassTwShared<LOG2M, NT> ltw{lps};
  for (int e = tid; e < sb / 4; e += NT)
    reinterpret_cast<float4 *>(A)[e] = make_float4(0.f, 0.f, 0.f, 0.f);

  // the running product in this thread's slots; the spectrum of FCS_d(T) in
  // the same slots (the q = 0 slot packs two reals) is read where it is first
  // used, since spectrum_kernel may still be running before
  float2 p[EPS][2][RL], X[EPS][2][RL];
  auto spec_at = [&](int e, int bb, int r) {
    const bool live = LPs::SLOTS % NT == 0 || tid + e * NT < LPs::SLOTS;
    const int q = live ? last_pass_index<LOG2M, NT>(e, bb, r) : 1;
    return live ? (q == 0 ? make_float2(__ldcg(&sd[0].x), __ldcg(&sd[M].x)) : __ldcg(sd + q))
                : make_float2(0.f, 0.f);
  };
  auto spec_to_p = [&] {
    griddep_wait();
#pragma unroll
    for (int e = 0; e < EPS; ++e)
#pragma unroll
      for (int bb = 0; bb < 2; ++bb)
#pragma unroll
        for (int r = 0; r < RL; ++r) p[e][bb][r] = spec_at(e, bb, r);
  };
  bool first = true;

  for (int n = 0; n < a.m.N; ++n) {
    if (!all && n == a.free_mode) continue;
    __syncthreads();
    const int32_t *hn = a.h + d * a.m.ldh + a.m.off[n];
    const int8_t *sn = a.s + d * a.m.ldh + a.m.off[n];
    const float *vn = a.vec[n] + b * a.m.I[n];
    for (int64_t i = tid; i < a.m.I[n]; i += NT) {
      float v = __ldg(vn + i);
      if (__ldg(sn + i) < 0) v = -v;
      const int hb = __ldg(hn + i);
      if (unsigned(hb) < unsigned(sb)) atomicAdd(A + hb, v);
    }
    rfft_to_slots<LOG2M, NT>(A, sb, B, tws, ltw, X);
    if (first && !all) spec_to_p();
#pragma unroll
    for (int e = 0; e < EPS; ++e)
#pragma unroll
      for (int bb = 0; bb < 2; ++bb)
#pragma unroll
        for (int r = 0; r < RL; ++r) {
          const bool packed = bb == 0 && r == 0 && tid + e * NT == 0;
          if (all && first)
            p[e][bb][r] = X[e][bb][r];
          else
            p[e][bb][r] = all ? slot_mul(p[e][bb][r], X[e][bb][r], packed)
                              : slot_mulconj(p[e][bb][r], X[e][bb][r], packed);
        }
    first = false;
  }
  if (first && !all) spec_to_p();                 // FREE of order 1
  griddep_launch();

  if (all) {
    griddep_wait();
    // sum_{k<P} conj(F_T[k]) Y[k]: the packed q = 0 slot holds the real bins
    // 0 and M (weight 1); every other bin q in (0, M) appears twice
    float part = 0.f;
#pragma unroll
    for (int e = 0; e < EPS; ++e) {
      if (LPs::SLOTS % NT != 0 && tid + e * NT >= LPs::SLOTS) continue;
#pragma unroll
      for (int bb = 0; bb < 2; ++bb)
#pragma unroll
        for (int r = 0; r < RL; ++r) {
          const bool packed = bb == 0 && r == 0 && tid + e * NT == 0;
          const float2 f = spec_at(e, bb, r);
          const float dot = f.x * p[e][bb][r].x + f.y * p[e][bb][r].y;
          part += packed ? dot : 2.f * dot;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((tid & 31) == 0) red[tid >> 5] = part;
    __syncthreads();
    if (tid == 0) {
      float t = 0.f;
      for (int w = 0; w < NT / 32; ++w) t += red[w];
      a.raw[b * a.D + d] = t / float(2 * M);
    }
    return;
  }

  if (a.kind == kBoth) {
    // p = F_T prod_{n != m} conj(F_n), so conj(p) F_m = conj(F_T) prod_n F_n:
    // T(v_1..v_N) is the Parseval sum of Re(conj(p) F_m) over the free
    // mode's transform, taken before p goes into the inverse transform
    const int m = a.free_mode;
    __syncthreads();
    const int32_t *hn = a.h + d * a.m.ldh + a.m.off[m];
    const int8_t *sn = a.s + d * a.m.ldh + a.m.off[m];
    const float *vn = a.vec[m] + b * a.m.I[m];
    for (int64_t i = tid; i < a.m.I[m]; i += NT) {
      float v = __ldg(vn + i);
      if (__ldg(sn + i) < 0) v = -v;
      const int hb = __ldg(hn + i);
      if (unsigned(hb) < unsigned(sb)) atomicAdd(A + hb, v);
    }
    rfft_to_slots<LOG2M, NT>(A, sb, B, tws, ltw, X);
    float part = 0.f;
#pragma unroll
    for (int e = 0; e < EPS; ++e) {
      if (LPs::SLOTS % NT != 0 && tid + e * NT >= LPs::SLOTS) continue;
#pragma unroll
      for (int bb = 0; bb < 2; ++bb)
#pragma unroll
        for (int r = 0; r < RL; ++r) {
          const bool packed = bb == 0 && r == 0 && tid + e * NT == 0;
          const float dot = p[e][bb][r].x * X[e][bb][r].x + p[e][bb][r].y * X[e][bb][r].y;
          part += packed ? dot : 2.f * dot;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((tid & 31) == 0) red[tid >> 5] = part;
    __syncthreads();
    if (tid == 0) {
      float t = 0.f;
      for (int w = 0; w < NT / 32; ++w) t += red[w];
      a.raw_all[b * a.D + d] = t / float(2 * M);
    }
  }

  // FREE: inverse transform of the product, then gather at h_m(i)
  slots_to_conj_packed<LOG2M, NT>(B, p, tw);
  __syncthreads();
  block_fft<LOG2M, NT>(B, tw);
  const int m = a.free_mode;
  const int32_t *hm = a.h + d * a.m.ldh + a.m.off[m];
  const int8_t *sm = a.s + d * a.m.ldh + a.m.off[m];
  const int64_t Im = a.m.I[m];
  float *rawbd = a.raw + (b * a.D + d) * Im;
  const float sc = 1.0f / float(M);
  const float *bufr = reinterpret_cast<const float *>(B);
  for (int64_t i = tid; i < Im; i += NT) {
    const int pz = __ldg(hm + i);
    const float v = unsigned(pz) < unsigned(2 * M) ? bufr[real_off(pz)] : __int_as_float(0x7fc00000);
    const float z = (pz & 1) ? -v * sc : v * sc;
    rawbd[i] = __ldg(sm + i) < 0 ? -z : z;
  }
}

// ---------------------------------------------------------------- P = 16384
// contract_kernel on the row-pair engine: one CTA per (item b, sketch d), two
// to an SM (contract_kernel's registers and buffers leave room for one).  The
// running product is in tensor memory between transforms, at the scale that it
// has in contract_kernel: the spectra are halved on the way (the unpack leaves
// twice the values), or a product of N would run out of range 2^N earlier.
template <int NR>
__global__ void __launch_bounds__(pfft::Geo<NR>::NT, pfft::Geo<NR>::CTAS)
    contract_pair_kernel(ContractArgs a, const float2 *__restrict__ tw) {
  using Geo = pfft::Geo<NR>;
  using Lay = pfft::Smem<NR>;
  constexpr int NT = Geo::NT, M = Geo::M, HALF = M / 2, H = Geo::H;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint32_t slot;
  __shared__ float red[NT / 32];
  float4 *B = reinterpret_cast<float4 *>(smem + Lay::kB);
  const float2 *t0 = reinterpret_cast<float2 *>(smem + Lay::kT0);
  const float2 *t1 = reinterpret_cast<float2 *>(smem + Lay::kT1);
  const float2 *t2 = reinterpret_cast<float2 *>(smem + Lay::kT2);
  const float2 *t3 = reinterpret_cast<float2 *>(smem + Lay::kT3);
  float4 *A4 = reinterpret_cast<float4 *>(smem + Lay::kA);
  float *A = reinterpret_cast<float *>(A4);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t b = blockIdx.x;
  const int d = blockIdx.y, N = a.m.N, sb = a.sb;
  const int ra = (sb + 2 * NR - 1) / (2 * NR);
  const bool all = a.kind == FCS_CONTRACT_ALL, both = a.kind == kBoth;
  const float2 *sd = a.spec + d * int64_t(M + 1);
  const uint32_t tm = pfft::tmem_alloc<NR>(&slot);
  const uint32_t tp = pfft::tmem_mine<NR>(tm);
  const bool w0 = warp == Geo::WARPS - 1;            // the warp that has column 0
  pfft::fill_twiddles<NR>(smem, tw);
  for (int e = tid; e < H * ra; e += NT) A4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  // mode of transform k: those of the product in order, the free one last
  const int last = all ? N - 1 : both ? N - 1 : N - 2;
  auto mode_of = [&](int k) {
    return all ? k : k == N - 1 ? a.free_mode : k < a.free_mode ? k : k + 1;
  };
  auto scatter = [&](int n) {
    const int32_t *hn = a.h + d * a.m.ldh + a.m.off[n];
    const int8_t *sn = a.s + d * a.m.ldh + a.m.off[n];
    const float *vn = a.vec[n] + b * a.m.I[n];
#pragma unroll 4
    for (int64_t i = tid; i < a.m.I[n]; i += NT) {
      const float v = __ldg(vn + i);
      const int hb = __ldg(hn + i);
      if (unsigned(hb) < unsigned(sb))
        atomicAdd(A + pfft::a_index<NR>(hb, ra), __ldg(sn + i) < 0 ? -v : v);
    }
  };
  if (last >= 0) scatter(mode_of(0));
  __syncthreads();
  float2 p0 = make_float2(1.f, lane == 0 ? 1.f : 0.f);   // column 0's product
  const int i0 = lane & (NR - 1);
  float2 f0 = make_float2(0.f, 0.f);                 // column 0 of FCS_d(T)'s spectrum
  auto spec_wait = [&] {
    griddep_wait();
    f0 = i0 ? __ldcg(sd + 512 * i0) : make_float2(__ldcg(&sd[0].x), __ldcg(&sd[M].x));
    if (!all) p0 = f0;
  };
  float part = 0.f;                                  // of the Parseval sum
  // spectrum of FCS_d(T) at the bins of value i (0 .. 2H - 1) of pair c
  auto spec_at = [&](int c, int i) {
    const int bb = i < H ? 0 : 1, k = i < H ? i : (2 * H - i) % H;
    const float2 u = __ldcg(sd + pfft::bin_of<NR>(c, bb, k, 0));
    const float2 v = __ldcg(sd + pfft::bin_of<NR>(c, bb, k, 1));
    return pfft::C2{pfft::pk(u.x, v.x), pfft::pk(u.y, v.y)};
  };
  for (int k = 0; k <= last; ++k) {
    pfft::scatter_row_step<Geo::RPW, Geo::PAD>(A4 + warp * ra, Geo::WARPS * ra, ra,
                                               B + warp * Geo::RS, Geo::WARPS * Geo::RS, t0, t1);
    __syncthreads();
    const bool early = tid < NT / 2;
    if (k < last && early) scatter(mode_of(k + 1));
    // dot: the Parseval sum over this transform (no product is kept)
    const bool dot = (all || both) && k == N - 1;
    if (k == (all ? N - 1 : 0)) spec_wait();         // first use of the spectrum
    if (w0) {
      float2 x = pfft::column0<NR>(B, t3);
      x = make_float2(0.5f * x.x, 0.5f * x.y);
      if (dot) {
        const float2 y = all ? slot_mul(p0, x, lane == 0) : x;
        const float2 g = all ? f0 : p0;
        if (lane < NR) part += (lane ? 2.f : 1.f) * (g.x * y.x + g.y * y.y);
      } else {
        p0 = all ? slot_mul(p0, x, lane == 0) : slot_mulconj(p0, x, lane == 0);
      }
    }
#pragma unroll 1
    for (int c = 0; c < Geo::NCP; ++c) {
      pfft::C2 xa[H], xc[H];
      pfft::column_step<NR, true>(B, t2, c, xa, xc);
      pfft::unpack<NR>(t2, c, xa, xc);
      const uint32_t o = tp + uint32_t(c) * (8 * H);
      __syncwarp();                                  // tensor-memory accesses are warp-wide
#pragma unroll
      for (int g = 0; g < 2 * H; g += 4) {
        pfft::Tm16 x;
        const bool load = k > 0;
        if (load) {
          pfft::tmem_ld16(o + 4 * g, x);
          pfft::tmem_wait_ld(x);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          pfft::C2 v = g < H ? xa[g + i] : xc[g - H + i];
          if (all) {
            if (load) v = pfft::cmul(pfft::tm_get(x, i), v);
          } else if (!dot) {
            const pfft::C2 y = load ? pfft::tm_get(x, i) : spec_at(c, g + i);
            v = pfft::cmul3(y, v.re, pfft::neg2(v.im), v.im);      // y conj(v)
          }
          if (dot) {
            const pfft::C2 f = all || !load ? spec_at(c, g + i) : pfft::tm_get(x, i);
            const pfft::f2x t = pfft::fma2(f.re, v.re, pfft::mul2(f.im, v.im));
            // (u = 256: its second column repeats the first)
            if (g < H || tid + c * NT != 255) part += 2.f * (pfft::lo(t) + pfft::hi(t));
          } else {
            pfft::tm_set(x, i, v);
          }
        }
        __syncwarp();
        if (!dot) pfft::tmem_st16(o + 4 * g, x);
      }
    }
    pfft::tmem_wait_st();
    if (k < last && !early) scatter(mode_of(k + 1));
    __syncthreads();
  }
  if (last < 0) spec_wait();                         // FREE of order 1
  griddep_launch();
  if (all || both) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0) red[warp] = part;
    __syncthreads();
    if (tid == 0) {
      float t = 0.f;
      for (int w = 0; w < NT / 32; ++w) t += red[w];
      (all ? a.raw : a.raw_all)[b * a.D + d] = t / float(2 * M);
    }
  }
  if (!all) {
    // FREE: the conj-packed product into B (every pair (q, M - q) is a
    // thread's), an inverse transform, then the gather at h_m(i)
    float *Bf = reinterpret_cast<float *>(B);
    auto put = [&](int m, float2 z) {
      float *p = Bf + pfft::b_index<NR>(m);
      p[0] = z.x;
      p[2] = z.y;
    };
#pragma unroll 1
    for (int c = 0; c < Geo::NCP; ++c) {
      const uint32_t o = tp + uint32_t(c) * (8 * H);
      pfft::Tm16 x[H / 2];
      __syncwarp();
      if (N > 1) {
#pragma unroll
        for (int g = 0; g < H / 2; ++g) pfft::tmem_ld16(o + 16 * g, x[g]);
#pragma unroll
        for (int g = 0; g < H / 2; ++g) pfft::tmem_wait_ld(x[g]);
      } else {                                       // no other mode: the sketch itself
#pragma unroll
        for (int i = 0; i < 2 * H; ++i) pfft::tm_set(x[i / 4], i % 4, spec_at(c, i));
      }
      const float2 wP = t2[Geo::LNR * 256 + tid + c * NT];
      const int u = tid + 1 + c * NT;
#pragma unroll
      for (int K = 0; K < H; ++K) {
        const int kc = H + (H - K) % H;
        const pfft::C2 va = pfft::tm_get(x[K / 4], K % 4), vc = pfft::tm_get(x[kc / 4], kc % 4);
        const float2 w = K == 0 ? wP : cmul(wP, unit64(K * 32 / NR));
        float2 cq, cm;
        const int q = u + 512 * K;
        pack_pair_conj_values_w(q, make_float2(pfft::lo(va.re), pfft::lo(va.im)),
                                make_float2(pfft::lo(vc.re), pfft::lo(vc.im)), w, cq, cm);
        put(q, cq);
        put(M - q, cm);
        const int r = q + HALF;
        pack_pair_conj_values_w(r, make_float2(pfft::hi(va.re), pfft::hi(va.im)),
                                make_float2(pfft::hi(vc.re), pfft::hi(vc.im)),
                                make_float2(w.y, -w.x), cq, cm);
        put(r, cq);
        put(M - r, cm);
      }
    }
    if (w0) {
      // lane i: X[512 i], paired with X[512 (NR - i)]
      float2 y;
      y.x = __shfl_sync(0xffffffffu, p0.x, (NR - i0) & (NR - 1));
      y.y = __shfl_sync(0xffffffffu, p0.y, (NR - i0) & (NR - 1));
      if (lane < NR) {
        float2 cq, cm;
        pack_pair_conj_values_w(lane, p0, y, t3[lane], cq, cm);
        put(512 * lane, lane == NR / 2 ? p0 : cq);
      }
    }
    __syncthreads();
    pfft::row_step<32, true, Geo::RPW, Geo::PAD>(B + warp * Geo::RS, Geo::WARPS * Geo::RS, 512,
                                                 B + warp * Geo::RS, Geo::WARPS * Geo::RS, t0, t1);
    __syncthreads();
    // z[m] in natural order over B once every column has been read
    float2 *Z = reinterpret_cast<float2 *>(B);
    pfft::C2 xa[Geo::NCP][H], xc[Geo::NCP][H];
#pragma unroll
    for (int c = 0; c < Geo::NCP; ++c) pfft::column_step<NR>(B, t2, c, xa[c], xc[c]);
    float2 z0 = make_float2(0.f, 0.f);
    if (w0) z0 = pfft::column0_complex<NR>(B, t3);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < Geo::NCP; ++c) {
      const int u = tid + 1 + c * NT, uc = 512 - u;
#pragma unroll
      for (int k = 0; k < H; ++k) {
        Z[u + 512 * k] = make_float2(pfft::lo(xa[c][k].re), pfft::lo(xa[c][k].im));
        Z[u + 512 * (k + H)] = make_float2(pfft::hi(xa[c][k].re), pfft::hi(xa[c][k].im));
        const int ql = (k == 0 ? NR - 1 : k + H - 1), qh = (k == 0 ? H - 1 : k - 1);
        Z[uc + 512 * ql] = make_float2(pfft::lo(xc[c][k].re), pfft::lo(xc[c][k].im));
        Z[uc + 512 * qh] = make_float2(pfft::hi(xc[c][k].re), pfft::hi(xc[c][k].im));
      }
    }
    if (w0 && lane < NR) Z[512 * lane] = z0;
    __syncthreads();
    const int m = a.free_mode;
    const int32_t *hm = a.h + d * a.m.ldh + a.m.off[m];
    const int8_t *sm = a.s + d * a.m.ldh + a.m.off[m];
    const int64_t Im = a.m.I[m];
    float *rawbd = a.raw + (b * a.D + d) * Im;
    const float sc = 1.0f / float(M);
    for (int64_t i = tid; i < Im; i += NT) {
      const int pz = __ldg(hm + i);
      const float v = unsigned(pz) < unsigned(2 * M) ? Bf[pz] : __int_as_float(0x7fc00000);
      const float z = (pz & 1) ? -v * sc : v * sc;
      rawbd[i] = __ldg(sm + i) < 0 ? -z : z;
    }
  }
  pfft::tmem_free<NR>(tm);
}

// raw [B][D][width] -> out [B][width] and, when out2 is given, raw2 [B][D] ->
// out2 [B].
template <int D>
__global__ void median_kernel(const float *raw, int64_t B, int64_t width, float *out,
                              const float *raw2, float *out2) {
  const int64_t total = B * width;
  griddep_wait();
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < total + (out2 ? B : 0);
       t += int64_t(gridDim.x) * blockDim.x) {
    const bool one = t < total;
    const int64_t w = one ? width : 1, e = one ? t : t - total;
    const int64_t b = e / w, i = e - b * w;
    const float *src = one ? raw : raw2;
    float v[D];
#pragma unroll
    for (int d = 0; d < D; ++d) v[d] = __ldcg(src + (b * D + d) * w + i);
    (one ? out : out2)[e] = median_inplace<D>(v);
  }
}

// P = 16384 has two kernels.  With more CTAs than SMs the row-pair engine is
// the faster one (order 3, 400^3, D = 5, both results: 64 items 64 us for 74,
// 1024 items 524 for 709); with fewer, one 512-thread CTA of contract_kernel
// has the shorter chain (10 items 33 us for 36).  At P = 8192 contract_kernel
// is as fast in large batches (1024 items 339 us for 324) and faster in small
// ones (10 items 23.5 us for 33.6).
template <int LOG2M>
int launch_contract(fcs_ctx *ctx, ContractArgs &a, int64_t Jt, bool need_spec,
                    cudaEvent_t spec_ready) {
  constexpr int NT = fft_threads(LOG2M);
  const int sb_spec = int((Jt + 3) / 4 * 4);
  const size_t smem1 = FftSmem<LOG2M>::bytes(sb_spec);
  const size_t smem2 = FftSmem<LOG2M>::bytes(a.sb);
  auto k1 = spectrum_kernel<LOG2M, NT>;
  auto k2 = contract_kernel<LOG2M, NT>;
  cudaError_t e = allow_smem(reinterpret_cast<const void *>(k1), smem1);
  if (e == cudaSuccess) e = allow_smem(reinterpret_cast<const void *>(k2), smem2);
  if (e != cudaSuccess) return check_cuda(ctx, e, "cudaFuncSetAttribute(contract)");
  if (need_spec) {
    k1<<<a.D, NT, smem1, ctx->stream>>>(a.fcsT, Jt, Jt, sb_spec, a.spec, ctx->twiddle);
    int rc = check_cuda(ctx, cudaGetLastError(), "spectrum_kernel");
    if (rc) return rc;
    if (spec_ready) {
      rc = check_cuda(ctx, cudaEventRecord(spec_ready, ctx->stream), "cudaEventRecord");
      if (rc) return rc;
    }
  }
  // Directly behind spectrum_kernel the transforms of the vectors start while
  // the D CTAs of the spectra still run (9 us of a chain of 42 at 64 items, P =
  // 8192, D = 5): the kernel waits where it first reads them.
  const bool overlap = need_spec && !spec_ready;
  const dim3 grid{unsigned(a.B), unsigned(a.D)};
  if constexpr (LOG2M == 13) {
    if (a.B * a.D > ctx->sm_count) {
      constexpr int NR = 16;
      const size_t smem3 = pfft::Smem<NR>::bytes((a.sb + 2 * NR - 1) / (2 * NR));
      auto k3 = contract_pair_kernel<NR>;
      e = allow_smem(reinterpret_cast<const void *>(k3), smem3);
      if (e != cudaSuccess) return check_cuda(ctx, e, "cudaFuncSetAttribute(contract)");
      return check_cuda(ctx, launch_dep(k3, grid, pfft::Geo<NR>::NT, smem3, ctx->stream, overlap,
                                        a, ctx->twiddle),
                        "contract_pair_kernel");
    }
  }
  return check_cuda(ctx, launch_dep(k2, grid, NT, smem2, ctx->stream, overlap, a, ctx->twiddle),
                    "contract_kernel");
}

// dep: the kernel before on the stream is the one that writes raw and raw2
int launch_median(fcs_ctx *ctx, int D, const float *raw, int64_t B, int64_t width, float *out,
                  const float *raw2, float *out2, bool dep) {
  const int64_t total = B * width + (out2 ? B : 0);
  cudaError_t e = cudaSuccess;
  int blocks = int((total + 255) / 256);
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  switch (D) {
#define FCS_MED_CASE(K) \
  case K:                                                                                   \
    e = launch_dep(median_kernel<K>, blocks, 256, 0, ctx->stream, dep, raw, B, width, out, \
                   raw2, out2);                                                            \
    break;
    FCS_MED_CASE(1) FCS_MED_CASE(2) FCS_MED_CASE(3) FCS_MED_CASE(4) FCS_MED_CASE(5)
    FCS_MED_CASE(6) FCS_MED_CASE(7) FCS_MED_CASE(8) FCS_MED_CASE(9) FCS_MED_CASE(10)
    FCS_MED_CASE(11) FCS_MED_CASE(12) FCS_MED_CASE(13) FCS_MED_CASE(14) FCS_MED_CASE(15)
    FCS_MED_CASE(16)
#undef FCS_MED_CASE
    default:
      return set_error(ctx, FCS_EINVAL, "D=%d outside [1,16]", D);
  }
  return check_cuda(ctx, e, "median_kernel");
}

}  // namespace

void spec_cache_invalidate(fcs_ctx *ctx, const void *p, size_t bytes) {
  fcs_spec_cache *c = ctx ? ctx->spec_cache : nullptr;
  if (!c) return;
  const char *lo = static_cast<const char *>(p);
  for (auto &x : c->e) {
    const char *k = reinterpret_cast<const char *>(x.key);
    if (k >= lo && k < lo + bytes) x.stale = true;
  }
}

void spec_cache_destroy(fcs_ctx *ctx) {
  fcs_spec_cache *c = ctx->spec_cache;
  if (!c) return;
  while (!c->e.empty()) spec_cache_erase(c, c->e.size() - 1);
  delete c;
  ctx->spec_cache = nullptr;
}

}  // namespace fcs

using namespace fcs;

extern "C" int fcs_cache_spectra(fcs_ctx *ctx, int enable) {
  if (!ctx) return FCS_EINVAL;
  ctx->err.clear();
  DeviceGuard g(ctx->device);
  if (!enable) spec_cache_destroy(ctx);
  ctx->cache_spectra = enable != 0;
  return FCS_OK;
}

extern "C" int fcs_forget(fcs_ctx *ctx, const void *ptr) {
  if (!ctx) return FCS_EINVAL;
  ctx->err.clear();
  fcs_spec_cache *c = ctx->spec_cache;
  if (!c || !ptr) return FCS_OK;
  for (auto &x : c->e)
    if (x.key == ptr) x.stale = true;        // recomputed on next use; no host wait
  return FCS_OK;
}

namespace {

// fcs_contract (kind ALL or FREE) and fcs_contract_both (kind kBoth: the FREE
// result in out_median / out_raw, the ALL result in out_all / out_all_raw).
int contract_call(fcs_ctx *ctx, int kind, int free_mode, int N, const int64_t *host_I,
                  const int32_t *host_J, int D, const float *fcsT, int64_t B,
                  const float *const *host_vecs, const int32_t *h, const int8_t *s,
                  int64_t ldh, float *out_median, float *out_raw, float *out_all,
                  float *out_all_raw) {
  if (!ctx) return FCS_EINVAL;
  ctx->err.clear();
  ContractArgs a{};
  int rc = make_modes(ctx, N, host_I, host_J, ldh, &a.m);
  if (rc) return rc;
  if (kind != FCS_CONTRACT_ALL && kind != FCS_CONTRACT_FREE && kind != kBoth)
    return set_error(ctx, FCS_EINVAL, "unknown contraction kind %d", kind);
  if (kind != FCS_CONTRACT_ALL && (free_mode < 0 || free_mode >= N))
    return set_error(ctx, FCS_EINVAL, "free_mode=%d outside [0,%d)", free_mode, N);
  if (D < 1 || D > kMaxD) return set_error(ctx, FCS_EINVAL, "D=%d outside [1,%d]", D, kMaxD);
  if (B < 1 || B > 65535) return set_error(ctx, FCS_EINVAL, "B=%lld outside [1,65535]", (long long)B);
  if (!fcsT || !host_vecs || !h || !s || !out_median || (kind == kBoth && !out_all))
    return set_error(ctx, FCS_EINVAL, "NULL pointer argument");
  for (int n = 0; n < N; ++n) {
    if (kind == FCS_CONTRACT_FREE && n == free_mode) {
      a.vec[n] = nullptr;
      continue;
    }
    if (!host_vecs[n]) return set_error(ctx, FCS_EINVAL, "vector %d is NULL", n);
    a.vec[n] = host_vecs[n];
  }
  const int log2p = ilog2_ceil(a.m.Jt) < kMinLog2P ? kMinLog2P : ilog2_ceil(a.m.Jt);
  if (log2p > kMaxLog2PBig)
    return set_error(ctx, FCS_EUNSUPPORTED, "Jt=%lld needs FFT length > %d",
                     (long long)a.m.Jt, 1 << kMaxLog2PBig);
  const int log2m = log2p - 1;
  const int64_t M = int64_t(1) << log2m;
  a.D = D;
  a.kind = kind;
  a.free_mode = free_mode;
  a.B = B;
  a.fcsT = fcsT;
  a.h = h;
  a.s = s;
  a.out = out_median;
  {
    int64_t jmax = 0;
    for (int n = 0; n < N; ++n) jmax = host_J[n] > jmax ? host_J[n] : jmax;
    a.sb = int((jmax + 3) / 4 * 4);
  }
  const int64_t width = kind == FCS_CONTRACT_ALL ? 1 : host_I[free_mode];
  const bool both = kind == kBoth;
  DeviceGuard g(ctx->device);
  bool hit = false;
  fcs_spec_cache::Entry *ent = spec_cache_get(ctx, fcsT, a.m.Jt, D, log2m, &hit);
  // the long-FFT path places its own spectrum buffer in the workspace; its
  // raw buffer must then come from a separate allocation owned by the context
  const bool big = log2p > kMaxLog2P;
  const size_t sbytes =
      (ent || big) ? 0 : (sizeof(float2) * size_t(D) * size_t(M + 1) + 255) & ~size_t(255);
  const size_t rbytes =
      out_raw ? 0 : (sizeof(float) * size_t(B) * D * size_t(width) + 255) & ~size_t(255);
  const size_t abytes = (both && !out_all_raw) ? sizeof(float) * size_t(B) * D : 0;
  if (big && rbytes + abytes) {
    rc = ensure_raw(ctx, rbytes + abytes);
    if (rc) return rc;
  }
  void *ws = nullptr;
  if (!big && sbytes + rbytes + abytes > 0) {
    rc = ensure_workspace(ctx, sbytes + rbytes + abytes, &ws);
    if (rc) return rc;
  }
  char *rbase = big ? reinterpret_cast<char *>(ctx->raw) : static_cast<char *>(ws) + sbytes;
  a.spec = ent ? ent->spec : static_cast<float2 *>(ws);
  a.raw = out_raw ? out_raw : reinterpret_cast<float *>(rbase);
  a.raw_all = !both ? nullptr
              : out_all_raw ? out_all_raw
                            : reinterpret_cast<float *>(rbase + rbytes);
  if (hit) {
    // the spectrum may have been written on another stream
    rc = check_cuda(ctx, cudaStreamWaitEvent(ctx->stream, ent->ready, 0), "cudaStreamWaitEvent");
    if (rc) return rc;
  }
  rc = FCS_EUNSUPPORTED;
  if (log2p > kMaxLog2P) {
    if (both) {
      // the long-FFT route runs the two contractions one after the other
      // (the second reuses the cached spectra when the cache is on)
      rc = big_contract(ctx, a.m, FCS_CONTRACT_ALL, free_mode, D, fcsT, B, a.vec, h, s,
                        ent ? ent->spec : nullptr, !hit, ent ? ent->ready : nullptr, a.raw_all,
                        log2p);
      if (!rc)
        rc = big_contract(ctx, a.m, FCS_CONTRACT_FREE, free_mode, D, fcsT, B, a.vec, h, s,
                          ent ? ent->spec : nullptr, ent == nullptr, nullptr, a.raw, log2p);
    } else {
      rc = big_contract(ctx, a.m, kind, free_mode, D, fcsT, B, a.vec, h, s,
                        ent ? ent->spec : nullptr, !hit, ent ? ent->ready : nullptr, a.raw,
                        log2p);
    }
  } else {
    FCS_DISPATCH_LOG2M(log2m, rc = launch_contract<L>(ctx, a, a.m.Jt, !hit,
                                                      ent ? ent->ready : nullptr));
  }
  if (rc) {
    if (ent && !hit) ent->stale = true;          // never computed
    return rc;
  }
  rc = launch_median(ctx, D, a.raw, B, width, out_median, a.raw_all, both ? out_all : nullptr,
                     !big);
  if (ent) {
    const int re =
        check_cuda(ctx, cudaEventRecord(ent->used, ctx->stream), "cudaEventRecord");
    if (!rc) rc = re;
  }
  return rc;
}

}  // namespace

extern "C" int fcs_contract(fcs_ctx *ctx, int kind, int free_mode, int N,
                            const int64_t *host_I, const int32_t *host_J, int D,
                            const float *fcsT, int64_t B, const float *const *host_vecs,
                            const int32_t *h, const int8_t *s, int64_t ldh,
                            float *out_median, float *out_raw) {
  if (kind != FCS_CONTRACT_ALL && kind != FCS_CONTRACT_FREE) {
    if (!ctx) return FCS_EINVAL;
    ctx->err.clear();
    return set_error(ctx, FCS_EINVAL, "unknown contraction kind %d", kind);
  }
  return contract_call(ctx, kind, free_mode, N, host_I, host_J, D, fcsT, B, host_vecs, h, s, ldh,
                       out_median, out_raw, nullptr, nullptr);
}

extern "C" int fcs_contract_both(fcs_ctx *ctx, int free_mode, int N, const int64_t *host_I,
                                 const int32_t *host_J, int D, const float *fcsT, int64_t B,
                                 const float *const *host_vecs, const int32_t *h,
                                 const int8_t *s, int64_t ldh, float *out_all, float *out_free,
                                 float *out_all_raw, float *out_free_raw) {
  return contract_call(ctx, kBoth, free_mode, N, host_I, host_J, D, fcsT, B, host_vecs, h, s,
                       ldh, out_free, out_free_raw, out_all, out_all_raw);
}
