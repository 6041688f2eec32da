// fcs_dense_items.cu -- fcs_sketch_dense for small tensors, eq. (FCS_asyn): one
// block per tensor of a batch.  The bin and sign of every entry and sketch
// depend on the hash tables alone, so a block works them out once, in shared
// memory, for all the tensors it takes, and with a whole tensor in one block
// its bins go to the output with plain stores: no clearing launch, no atomics
// on the output, no per-row tables.  dense_rows_kernel gives such a tensor a
// block of 768 threads of which a few warps have a row: 256 tensors of 7 x 7 x
// 32 at D = 5 took 53 us there with the clearing launch, 20 us here; bound by
// latency (tables, then one pass).
//
// Sums are exact, as there: the block knows its largest entry, 2^E above it,
// and rounds every entry once to a multiple of q = 2^(E - 30); the integer goes
// to two int32 bins, its lower 15 bits to one and the rest to the other, which
// at most 2^15 entries cannot overflow.  Where that rounding, q / sqrt(12),
// exceeds 1e-7 of the entries' geometric mean (which a few outliers hardly
// move; N(0,1) entries are 20 times below), one int32 bin takes the entries as
// multiples of 2^(E - 17) and the other, in FP32 with compare-and-swap
// atomics, what that leaves of them, so that large entries cost the small ones
// no digits (200 tensors of 64 x 64 with log-normal entries, D = 5: error 2.6e-8
// for 1.1e-7 with FP32 sums alone, 49 us for 43).
// Entries that are not finite, or too large or small for the powers of two, are
// added in FP32 as they are.
#include <algorithm>

#include "fcs_dense_items.cuh"

namespace fcs {
namespace {

constexpr int kNT = 256;
constexpr int kMaxEntries = 8192;         // per tensor

struct ItemArgs {
  int N, D, n, tot, Jt;
  int I[kMaxN], off[kMaxN], J[kMaxN];     // off: offset of a mode in a table row
  int64_t ldh, tbs, obs, nbatch;
  const float *T;
  const int32_t *h;
  const int8_t *s;
  float *out;
};

size_t items_smem(int D, int n, int tot, int Jt) {
  return 2 * sizeof(int) * size_t(D) * size_t(Jt) + sizeof(int) * size_t(D) * size_t(tot) +
         sizeof(uint16_t) * size_t(D) * size_t(n);
}

__global__ void __launch_bounds__(kNT) dense_items_kernel(ItemArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  int *hb = reinterpret_cast<int *>(smem);                 // [D][Jt]
  int *lb = hb + a.D * a.Jt;                               // [D][Jt]
  int *tab = lb + a.D * a.Jt;                              // [D][tot] hash << 1 | negative, -1
  uint16_t *bin = reinterpret_cast<uint16_t *>(tab + a.D * a.tot);   // [D][n] bin << 1 | negative
  float *lf = reinterpret_cast<float *>(lb);
  __shared__ float red[kNT / 32];
  __shared__ int exps[kNT / 32], nonzero[kNT / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < a.D * a.tot; e += kNT) {
    const int d = e / a.tot, k = e - d * a.tot;
    int n = 0;
    while (n + 1 < a.N && k >= a.off[n + 1]) ++n;
    const int v = a.h[d * a.ldh + k];
    tab[e] = unsigned(v) < unsigned(a.J[n]) ? (v << 1) | (a.s[d * a.ldh + k] < 0 ? 1 : 0) : -1;
  }
  for (int e = tid; e < 2 * a.D * a.Jt; e += kNT) hb[e] = 0;
  __syncthreads();
  for (int e = tid; e < a.n; e += kNT) {
    int idx[kMaxN], r = e;
    for (int n = a.N - 1; n >= 0; --n) {
      const int q = r / a.I[n];
      idx[n] = a.off[n] + r - q * a.I[n];
      r = q;
    }
    for (int d = 0; d < a.D; ++d) {
      int b = 0, neg = 0;
      bool ok = true;
      for (int n = 0; n < a.N; ++n) {
        const int t = tab[d * a.tot + idx[n]];
        ok = ok && t >= 0;
        b += t >> 1;
        neg ^= t & 1;
      }
      bin[d * a.n + e] = ok ? uint16_t((b << 1) | neg) : uint16_t(0xffff);
    }
  }
  __syncthreads();
  for (int64_t item = blockIdx.x; item < a.nbatch; item += gridDim.x) {
    const float *T = a.T + item * a.tbs;
    float m = 0.f;
    int ex = 0, nz = 0;                    // binary exponents (biased) of the entries that are not 0
    bool fin = true;
    for (int e = tid; e < a.n; e += kNT) {
      const float x = fabsf(__ldg(T + e));
      fin = fin && x <= 3.4e38f;           // false for NaN and Inf
      m = fmaxf(m, x);
      ex += __float_as_int(x) >> 23;
      nz += x > 0.f;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      ex += __shfl_xor_sync(0xffffffffu, ex, o);
      nz += __shfl_xor_sync(0xffffffffu, nz, o);
    }
    if (lane == 0) {
      red[warp] = m;
      exps[warp] = ex;
      nonzero[warp] = nz;
    }
    const bool finite = __syncthreads_and(fin);
    m = 0.f;
    ex = nz = 0;
#pragma unroll
    for (int k = 0; k < kNT / 32; ++k) {
      m = fmaxf(m, red[k]);
      ex += exps[k];
      nz += nonzero[k];
    }
    int E = 0;
    frexpf(m, &E);                                         // |x| < 2^E
    E -= 30;
    // log2 of both sides of q / sqrt(12) <= 1e-7 * geometric mean
    const bool fixed = finite && nz > 0 && E > -120 && E < 95 &&
                       float(E) - 1.8f <= float(ex) / float(nz) - 127.f - 23.3f;
    // otherwise the two parts of every entry, or no integers at all
    const bool parts = !fixed && finite && nz > 0 && E > -120 && E < 95;
    if (parts) E += 13;
    const float q = fixed || parts ? ldexpf(1.f, E) : 1.f;
    const float inv_q = fixed || parts ? ldexpf(1.f, -E) : 1.f;
    for (int e = tid; e < a.n; e += kNT) {
      const float x = __ldg(T + e);
      if (fixed) {
        const int xi = __float2int_rn(x * inv_q);
        for (int d = 0; d < a.D; ++d) {
          const unsigned t = bin[d * a.n + e];
          if (t == 0xffffu) continue;
          const int v = (t & 1) ? -xi : xi;
          atomicAdd(&hb[d * a.Jt + (t >> 1)], v >> 15);
          atomicAdd(&lb[d * a.Jt + (t >> 1)], v & 0x7fff);
        }
      } else {
        // (|xi| <= 2^17: 2^13 entries of a bin stay below 2^31; r is exact)
        const int xi = parts ? __float2int_rn(x * inv_q) : 0;
        const float r = parts ? fmaf(-q, float(xi), x) : x;
        for (int d = 0; d < a.D; ++d) {
          const unsigned t = bin[d * a.n + e];
          if (t == 0xffffu) continue;
          if (xi) atomicAdd(&hb[d * a.Jt + (t >> 1)], (t & 1) ? -xi : xi);
          if (r != 0.f) atomicAdd(&lf[d * a.Jt + (t >> 1)], (t & 1) ? -r : r);
        }
      }
    }
    __syncthreads();
    float *out = a.out + item * a.obs;
    for (int e = tid; e < a.D * a.Jt; e += kNT) {
      // (a 46-bit integer is exact in FP64; q is a power of two)
      out[e] = fixed   ? float((double(hb[e]) * 32768. + double(lb[e])) * double(q))
               : parts ? float(double(hb[e]) * double(q) + double(lf[e]))
                       : lf[e];
      hb[e] = 0;
      lb[e] = 0;
    }
    __syncthreads();
  }
}

}  // namespace

int dense_items(fcs_ctx *ctx, int N, const int64_t *I, const int64_t *stride, const int64_t *off,
                const int32_t *J, int64_t ldh, int64_t Jt, int D, const float *T, const int32_t *h,
                const int8_t *s, float *out, int64_t nbatch, int64_t tbs, int64_t obs, bool *done) {
  *done = false;
  ItemArgs a{};
  int64_t n = 1, tot = 0;
  for (int k = N - 1; k >= 0; --k) {
    if (I[k] > 1 && stride[k] != n) return FCS_OK;         // densely packed tensors only
    n *= I[k];
    if (n > kMaxEntries) return FCS_OK;
  }
  // modes in table order (the caller's order may differ: then off is not ascending)
  for (int k = 0; k < N; ++k) {
    if (off[k] != tot) return FCS_OK;
    tot += I[k];
    a.I[k] = int(I[k]);
    a.off[k] = int(off[k]);
    a.J[k] = J[k];
  }
  // Bins of 15 bits.  A tensor in one block is a long chain, so it takes enough
  // tensors to give every SM one (us here / by row blocks; 256 tensors of 512
  // entries at D = 5 8 / 22, 1764 at D = 10 35 / 62, 4096 at D = 5 43 / 155, 8000
  // at D = 1 36 / 80; but 32 tensors of 4096 at D = 5 33 / 29, 16384 at D = 1 60 /
  // 15) unless the chain is short (one tensor of 512 at D = 5 6.7 / 8.6, at D = 10
  // 10 / 10 to 20, of 1764 at D = 10 27 / 12).
  if (Jt > 32767 || (n * D > 6144 && nbatch < ctx->sm_count)) return FCS_OK;
  const size_t smem = items_smem(D, int(n), int(tot), int(Jt));
  if (smem > 100 * 1024) return FCS_OK;
  a.N = N;
  a.D = D;
  a.n = int(n);
  a.tot = int(tot);
  a.Jt = int(Jt);
  a.ldh = ldh;
  a.tbs = tbs;
  a.obs = obs;
  a.nbatch = nbatch;
  a.T = T;
  a.h = h;
  a.s = s;
  a.out = out;
  const cudaError_t e = allow_smem(reinterpret_cast<const void *>(dense_items_kernel), smem);
  if (e != cudaSuccess) return check_cuda(ctx, e, "cudaFuncSetAttribute(dense_items)");
  const int per_sm = std::max(1, std::min(8, int(size_t(233472) / (smem + 2048))));
  const int64_t blocks = std::min<int64_t>(nbatch, int64_t(ctx->sm_count) * per_sm);
  dense_items_kernel<<<unsigned(blocks), kNT, smem, ctx->stream>>>(a);
  *done = true;
  return check_cuda(ctx, cudaGetLastError(), "dense_items_kernel");
}

}  // namespace fcs
