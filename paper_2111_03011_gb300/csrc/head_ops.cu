// What is done with a finished head H[L][2^h] (complex128): amplitude lookup,
// norms, XEB sums and the group samplers.
//
// GB300 has little FP64 arithmetic (about two FP64 lanes per clock and SM), so
// the kernels that reduce a whole head are bound by FP64 instructions long
// before HBM; they are written to spend few of them per amplitude, and none
// where an FP32 estimate with a proven error settles a comparison.
//
// Results that the host waits for (norm, XEB sums, the first missing index, the
// plan's status word) are stored by the kernels into a HeadReport in mapped
// host memory, so that a call is its kernels and one synchronisation, with no
// copies of a few bytes around them.
//
// Whole calls, before (a warp scan per 32 members in every kernel, status words
// and results by copies) and now; a launch and a synchronisation take 14 us:
//   amplitudes, 65,536 of 64 groups, pinned host in and out    54 ->  26 us
//   norm with group norms, 64 groups of 1,024                  74 ->  31 us
//   norm, 65,536 groups of 64                                 123 ->  48 us
//   10,000 exact draws, 64 groups of 1,024                    362 ->  37 us
//   65,536 exact draws, 65,536 groups of 64                   198 ->  39 us
//   XEB of 65,536 samples, 65,536 groups                       63 ->  37 us
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"

namespace tn {

static constexpr int kSMs = 152;

// The plan's status word (a bounded wait of a contraction that gave up) as it
// stands when this kernel runs, for the host to read after it synchronises.
__device__ __forceinline__ void report_word(HeadReport* rep, const unsigned int* plan_status) {
  if (rep && plan_status && blockIdx.x == 0 && threadIdx.x == 0) rep->word = *plan_status;
}

// ---------------------------------------------------------------------- K7
// Index into H of bitstring b (its tail's group by binary search over the
// sorted tails, its open bits gathered), or -1.
__device__ __forceinline__ int64_t head_index(uint64_t b, int h, const uint64_t* __restrict__ keys,
                                              const uint32_t* __restrict__ groups, int64_t n_keys,
                                              uint64_t tail_mask, const int* __restrict__ open_q) {
  const uint64_t key = b & tail_mask;
  int64_t lo = 0, hi = n_keys;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (__ldg(keys + mid) < key) lo = mid + 1; else hi = mid;
  }
  if (lo >= n_keys || __ldg(keys + lo) != key) return -1;
  int64_t mu = 0;
  for (int j = 0; j < h; ++j) mu |= (int64_t)((b >> __ldg(open_q + j)) & 1ULL) << j;
  return ((int64_t)__ldg(groups + lo) << h) + mu;
}

// With seg_end (n_seg cumulative ends of merged requests), a missing key i of
// segment j records its index within the segment in status[j]; otherwise
// status[0] receives the smallest missing index.  `status` may be mapped host
// memory: it is touched for missing keys only.
__global__ void k_amplitudes(const double2* __restrict__ H, int h, const uint64_t* __restrict__ keys,
                             const uint32_t* __restrict__ groups, int64_t n_keys, uint64_t tail_mask,
                             const int* __restrict__ open_q, const uint64_t* __restrict__ bits, int64_t n, void* out,
                             int dtype, unsigned long long* status, const int64_t* __restrict__ seg_end, int n_seg,
                             HeadReport* rep, const unsigned int* plan_status) {
  report_word(rep, plan_status);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t at = head_index(bits[i], h, keys, groups, n_keys, tail_mask, open_q);
    double2 v = make_double2(0.0, 0.0);
    if (at >= 0) {
      v = H[at];
    } else if (seg_end) {
      int j = 0;
      while (j < n_seg - 1 && i >= seg_end[j]) ++j;
      atomicMin(status + j, (unsigned long long)(i - (j ? seg_end[j - 1] : 0)));
    } else {
      atomicMin_system(status, (unsigned long long)i);
    }
    if (dtype == 1) ((double2*)out)[i] = v;
    else ((float2*)out)[i] = make_float2((float)v.x, (float)v.y);
  }
}

cudaError_t launch_amplitudes(const double2* H, int h, const uint64_t* keys, const uint32_t* groups, int64_t n_keys,
                              uint64_t tail_mask, const int* open_q, const uint64_t* bits, int64_t n, void* out,
                              int dtype, unsigned long long* status, cudaStream_t s, const int64_t* seg_end,
                              int n_seg, HeadReport* rep, const unsigned int* plan_status) {
  if (n <= 0) return cudaSuccess;
  const int64_t grid = std::min<int64_t>((n + 255) / 256, (int64_t)kSMs * 8);
  k_amplitudes<<<(unsigned)grid, 256, 0, s>>>(H, h, keys, groups, n_keys, tail_mask, open_q, bits, n, out, dtype,
                                              status, seg_end, n_seg, rep, plan_status);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------- K5
// Norms.  Two FP64 instructions per amplitude (fused multiply-adds into two
// running sums per lane): 2.4 per 32 amplitudes and lane with the reductions of
// a group of 64, where a warp scan per 32 amplitudes took nine.
//   narrow groups (up to 512 members): 2^g lanes per group, at least eight
//     members a lane, several groups per warp;
//   wide groups: a block per unit, a group cut into 2^seg units where there
//     are fewer groups than the chip has room for.
// Z[g] (or the units' sums) and each block's total go to memory; k_norm_final
// adds them in index order, so the result depends on the sizes alone.
__global__ void __launch_bounds__(256) k_norm_narrow(const double2* __restrict__ H, int64_t L, int h, int lanes_log2,
                                                     double* __restrict__ Z, double* __restrict__ part) {
  __shared__ double wsum[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int G = 1 << lanes_log2, per = 1 << (h - lanes_log2);     // lanes per group, members per lane
  const int sub = lane & (G - 1);
  double total = 0.0;
  const int64_t per_warp = 32 >> lanes_log2;
  for (int64_t g0 = ((int64_t)blockIdx.x * 8 + warp) * per_warp; g0 < L; g0 += (int64_t)gridDim.x * 8 * per_warp) {
    const int64_t g = g0 + (lane >> lanes_log2);
    double a = 0.0, b = 0.0;
    if (g < L) {
      const double2* p = H + (g << h) + sub;
#pragma unroll 8
      for (int j = 0; j < per; ++j) {
        const double2 v = __ldg(p + (int64_t)j * G);
        a = fma(v.x, v.x, a);
        b = fma(v.y, v.y, b);
      }
    }
    a += b;
    for (int d = 1; d < G; d <<= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
    if (sub == 0 && g < L) {
      Z[g] = a;
      total += a;
    }
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) total += __shfl_xor_sync(0xffffffffu, total, d);
  if (lane == 0) wsum[warp] = total;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += wsum[w];
    part[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(256) k_norm_wide(const double2* __restrict__ H, int64_t L, int h, int seg_log2,
                                                   double* __restrict__ Z, double* __restrict__ part,
                                                   double* __restrict__ unit) {
  __shared__ double wsum[8];
  const int64_t n = 1LL << (h - seg_log2);                        // members of a unit
  double total = 0.0;
  for (int64_t u = blockIdx.x; u < L << seg_log2; u += gridDim.x) {
    const double2* p = H + u * n;
    double a = 0.0, b = 0.0;
#pragma unroll 4
    for (int64_t i = threadIdx.x; i < n; i += 256) {
      const double2 v = __ldg(p + i);
      a = fma(v.x, v.x, a);
      b = fma(v.y, v.y, b);
    }
    a += b;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < 8; ++w) t += wsum[w];
      if (seg_log2) unit[u] = t; else Z[u] = t;
      total += t;
    }
  }
  if (threadIdx.x == 0) part[blockIdx.x] = total;
}

// One block: N = sum of the blocks' totals and, with units, Z[g] = sum of its
// units, each in index order per thread.  n_sums = 2: the two XEB sums instead.
__global__ void __launch_bounds__(1024) k_final_sums(const double* __restrict__ part, int nb, int n_sums,
                                                     const double* __restrict__ unit, int64_t L, int seg_log2,
                                                     double* __restrict__ Z, double* out, HeadReport* rep,
                                                     const unsigned int* plan_status, double* host_Z) {
  __shared__ double w[32];
  report_word(rep, plan_status);
  if (seg_log2)
    for (int64_t g = threadIdx.x; g < L; g += blockDim.x) {
      double t = 0.0;
      for (int64_t s = 0; s < 1LL << seg_log2; ++s) t += unit[(g << seg_log2) + s];
      Z[g] = t;
      if (host_Z) host_Z[g] = t;
    }
  else if (host_Z)
    for (int64_t g = threadIdx.x; g < L; g += blockDim.x) host_Z[g] = Z[g];
  for (int q = 0; q < n_sums; ++q) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) acc += part[(int64_t)q * nb + i];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
      double v = threadIdx.x < (blockDim.x >> 5) ? w[threadIdx.x] : 0.0;
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
      if (threadIdx.x == 0) {
        if (out) out[q] = v;
        if (rep) rep->sum[q] = v;
      }
    }
  }
}

cudaError_t launch_group_norms(const double2* H, int64_t L, int h, double* Z, double* N, double* scratch,
                               cudaStream_t s, HeadReport* rep, const unsigned int* plan_status, double* host_Z) {
  double* part = scratch;                      // kHeadParts block totals, then kHeadParts units
  double* unit = scratch + kHeadParts;
  int nb, seg = 0;
  if (h <= 9) {
    const int lanes = h <= 3 ? 0 : std::min(5, h - 3);
    const int64_t per_block = 8 * (32 >> lanes);
    nb = (int)std::min<int64_t>((L + per_block - 1) / per_block, kHeadParts);
    k_norm_narrow<<<(unsigned)nb, 256, 0, s>>>(H, L, h, lanes, Z, part);
  } else {
    // units of at least 1,024 members until every SM has a few
    while ((L << seg) * 2 <= kHeadParts && h - seg > 10) ++seg;
    nb = (int)std::min<int64_t>(L << seg, kHeadParts);
    k_norm_wide<<<(unsigned)nb, 256, 0, s>>>(H, L, h, seg, Z, part, unit);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_final_sums<<<1, 1024, 0, s>>>(part, nb, 1, unit, L, seg, Z, N, rep, plan_status, host_Z);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------- K9
// XEB: for every sample, w = |H[sample]|^2; the blocks' sums of w and of log w
// (FP64), then one block adds them.  Looking the amplitudes up here saves
// writing and reading them.
__global__ void __launch_bounds__(256) k_xeb(const double2* __restrict__ H, int h, const uint64_t* __restrict__ keys,
                                             const uint32_t* __restrict__ groups, int64_t n_keys, uint64_t tail_mask,
                                             const int* __restrict__ open_q, const uint64_t* __restrict__ samples,
                                             int64_t n, double* __restrict__ part, unsigned long long* status) {
  __shared__ double s1[8], s2[8];
  double p = 0.0, lp = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t at = head_index(samples[i], h, keys, groups, n_keys, tail_mask, open_q);
    if (at < 0) {
      atomicMin_system(status, (unsigned long long)i);
      continue;
    }
    const double2 v = H[at];
    const double w = v.x * v.x + v.y * v.y;
    p += w;
    lp += log(w);
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    p += __shfl_xor_sync(0xffffffffu, p, d);
    lp += __shfl_xor_sync(0xffffffffu, lp, d);
  }
  if ((threadIdx.x & 31) == 0) {
    s1[threadIdx.x >> 5] = p;
    s2[threadIdx.x >> 5] = lp;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t1 = 0.0, t2 = 0.0;
    for (int w = 0; w < 8; ++w) {
      t1 += s1[w];
      t2 += s2[w];
    }
    part[blockIdx.x] = t1;
    part[gridDim.x + blockIdx.x] = t2;
  }
}

cudaError_t launch_xeb(const double2* H, int h, const uint64_t* keys, const uint32_t* groups, int64_t n_keys,
                       uint64_t tail_mask, const int* open_q, const uint64_t* samples, int64_t n, double* scratch,
                       HeadReport* rep, cudaStream_t s) {
  const int nb = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, kHeadParts));
  k_xeb<<<(unsigned)nb, 256, 0, s>>>(H, h, keys, groups, n_keys, tail_mask, open_q, samples, n, scratch,
                                     &rep->missing);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_final_sums<<<1, 1024, 0, s>>>(scratch, nb, 2, nullptr, 0, 0, nullptr, nullptr, rep, nullptr, nullptr);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------- K6
// Philox-4x32-10 (Salmon et al., SC'11): multipliers 0xD2511F53, 0xCD9E8D57,
// Weyl key increments 0x9E3779B9, 0xBB67AE85, ten rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    if (r != 9) { k.x += 0x9E3779B9u; k.y += 0xBB67AE85u; }
  }
  return c;
}

__device__ __forceinline__ double u53(uint32_t lo, uint32_t hi) {
  const uint64_t x = ((uint64_t)hi << 32) | lo;
  return (double)(x >> 11) * 0x1.0p-53;
}

// |h|^2 with each operation rounded to nearest (no fused multiply-add), so
// that weights and the comparisons built on them are reproducible bit by bit.
__device__ __forceinline__ double weight_rn(double2 v) { return __dadd_rn(__dmul_rn(v.x, v.x), __dmul_rn(v.y, v.y)); }

__device__ __forceinline__ double warp_inclusive_scan(double v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const double u = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += u;
  }
  return v;
}

// The sampler's prefix sums.  A group's members are taken in chunks of 32: the
// prefix inside a chunk is the warp scan above, and carry[c] is the sum of the
// chunks before c, added one chunk at a time.  A scan's last value is a balanced
// tree over adjacent pairs, which a butterfly adds in the same pairs; eight
// chunks go through one butterfly at a time (after its first three steps
// a lane holds one chunk), 9 additions instead of 40, with the same bits.
// H: from the first of the n_groups groups on.
__global__ void __launch_bounds__(256) k_group_prefix(const double2* __restrict__ H, int h, int64_t n_groups,
                                                      double* __restrict__ carry) {
  constexpr int kPiece = 1024;                 // chunks per pass through shared memory
  __shared__ double tot[kPiece];
  __shared__ double run;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t l = 1LL << h, nch = (l + 31) >> 5;
  for (int64_t g = blockIdx.x; g < n_groups; g += gridDim.x) {
    double* out = carry + g * (nch + 1);
    if (threadIdx.x == 0) {
      run = 0.0;
      out[0] = 0.0;
    }
    for (int64_t c0 = 0; c0 < nch; c0 += kPiece) {
      const int m = (int)min((int64_t)kPiece, nch - c0);
      __syncthreads();
      for (int b = warp * 8; b < m; b += 64) {
        double w[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int64_t i = (c0 + b + j) * 32 + lane;
          w[j] = i < l ? weight_rn(H[(g << h) + i]) : 0.0;
        }
#pragma unroll
        for (int st = 0; st < 3; ++st) {
          const bool up = (lane >> st) & 1;
#pragma unroll
          for (int j = 0; j < (4 >> st); ++j) {
            const double keep = up ? w[2 * j + 1] : w[2 * j], send = up ? w[2 * j] : w[2 * j + 1];
            w[j] = keep + __shfl_xor_sync(0xffffffffu, send, 1 << st);
          }
        }
        w[0] += __shfl_xor_sync(0xffffffffu, w[0], 8);
        w[0] += __shfl_xor_sync(0xffffffffu, w[0], 16);
        if (lane < 8 && b + lane < m) tot[b + lane] = w[0];
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        double r = run;
#pragma unroll 8
        for (int c = 0; c < m; ++c) {
          r += tot[c];
          tot[c] = r;
        }
        run = r;
      }
      __syncthreads();
      for (int c = threadIdx.x; c < m; c += 256) out[c0 + c + 1] = tot[c];
    }
    __syncthreads();
  }
}

// The first member whose prefix exceeds t, by the chunk scans from chunk c0 on
// (the sampler's definition); l - 1 if none does.
__device__ __forceinline__ int64_t scan_from(const double2* __restrict__ Hg, int64_t l, int64_t c0, double carry,
                                             double t) {
  const int lane = threadIdx.x & 31;
  for (int64_t c = c0 * 32; c < l; c += 32) {
    const double w = (c + lane < l) ? weight_rn(Hg[c + lane]) : 0.0;
    const double s = warp_inclusive_scan(w);
    const unsigned ball = __ballot_sync(0xffffffffu, (c + lane < l) && (carry + s > t));
    if (ball) return c + __ffs(ball) - 1;
    carry += __shfl_sync(0xffffffffu, s, 31);
  }
  return l - 1;
}

__device__ __forceinline__ int64_t scan_total_and_pick(const double2* __restrict__ Hg, int64_t l, double u_pick) {
  const int lane = threadIdx.x & 31;
  double Z = 0.0;
  for (int64_t c = 0; c < l; c += 32) {
    const double s = warp_inclusive_scan((c + lane < l) ? weight_rn(Hg[c + lane]) : 0.0);
    Z += __shfl_sync(0xffffffffu, s, 31);
  }
  if (Z > 0.0) return scan_from(Hg, l, 0, 0.0, u_pick * Z);
  const int64_t mu = (int64_t)(u_pick * (double)l);
  return mu >= l ? l - 1 : mu;
}

// The group's tail with the open bits of mu (lane j places bit j).
__device__ __forceinline__ uint64_t bitstring_of(const SampleParams& p, int64_t g, int64_t mu) {
  const int lane = threadIdx.x & 31;
  uint64_t b = lane < p.h ? (uint64_t)((mu >> lane) & 1) << p.open_q[lane] : 0ULL;
  const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)b), hi = __reduce_or_sync(0xffffffffu, (uint32_t)(b >> 32));
  return (p.tails[g] & ~p.open_mask) | ((uint64_t)hi << 32) | lo;
}

// Sample j of the launch and its group: sample i is drawn from group i mod L; with
// a window of groups the launch takes those samples whose group is in it.
__device__ __forceinline__ int64_t sample_of(const SampleParams& p, int64_t j, int64_t& g) {
  if (p.win == 0) {
    g = j % p.L;
    return j;
  }
  const int64_t round = j / p.win;
  g = p.g0 + (j - round * p.win);
  return round * p.L + g;
}

__device__ __forceinline__ uint64_t uniform_string(const SampleParams& p, int64_t i, uint2 key) {
  const uint64_t full = p.n_qubits >= 64 ? ~0ULL : ((1ULL << p.n_qubits) - 1);
  const uint4 q = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)((uint64_t)i >> 32), 1u, 0u), key);
  return ((((uint64_t)q.y) << 32) | q.x) & full;
}

// Exact draw with the groups' prefix sums at hand (wide groups, or several
// samples per group): a warp per sample finds the chunk by a 32-way search over
// the carries and scans that chunk.  A lane of an earlier chunk may exceed t
// by rounding alone (its scan and the chunk's total are different trees, a few
// ulp apart), so the scan starts at the first carry above t (1 - 2^-40).
__global__ void __launch_bounds__(256) k_sample_prefix(SampleParams p) {
  report_word(p.rep, p.plan_status);
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t l = 1LL << p.h, nch = (l + 31) >> 5;
  const uint2 key = make_uint2((uint32_t)p.seed, (uint32_t)(p.seed >> 32));
  for (int64_t j = warp; j < p.m; j += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    int64_t g;
    const int64_t i = sample_of(p, j, g);
    const uint4 r = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)((uint64_t)i >> 32), 0u, 0u), key);
    if (p.mix > 0.0 && u53(r.x, r.y) < p.mix) {
      if (lane == 0) p.out[i] = uniform_string(p, i, key);
      continue;
    }
    const double u_pick = u53(r.z, r.w);
    const double* __restrict__ cr = p.carry + (g - p.g0) * (nch + 1);
    const double Z = cr[nch];
    int64_t mu;
    if (Z > 0.0) {
      const double t = u_pick * Z, low = t * (1.0 - 0x1.0p-40);
      int64_t lo = 0, hi = nch;                 // the first chunk with carry[c + 1] > low is in [lo, hi)
      bool found = true;
      while (hi - lo > 1 && found) {
        const int64_t step = (hi - lo + 31) >> 5;
        const int64_t c = min(lo + (lane + 1) * step, hi);
        const unsigned ball = __ballot_sync(0xffffffffu, cr[c] > low);
        found = ball != 0;
        const int f = __ffs(ball) - 1;
        const int64_t base = lo;
        lo = base + f * step;
        hi = min(base + (f + 1) * step, hi);
      }
      mu = found ? scan_from(p.H + (g << p.h), l, lo, cr[lo], t) : l - 1;
    } else {
      mu = (int64_t)(u_pick * (double)l);
      if (mu >= l) mu = l - 1;
    }
    const uint64_t s = bitstring_of(p, g, mu);
    if (lane == 0) p.out[i] = s;
  }
}

// A double as a float of value x 2^shift, by its bits (a conversion would run
// on the FP64 pipe): truncated to 24 bits, 0 below the float range, infinity
// above it and for infinities and NaN.  The sign is dropped.
__device__ __forceinline__ float abs_as_float(double x, int shift) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ff);
  const int f = e - 1023 + 127 + shift;
  const uint32_t m = ((hi & 0xfffffu) << 3) | (lo >> 29);
  if (f <= 0) return 0.0f;
  if (f >= 255 || e == 0x7ff) return __int_as_float(0x7f800000);
  return __uint_as_float(((uint32_t)f << 23) | m);
}

// Exact draw from narrow groups (up to 32 NCH members), one pass over a
// group.  The draw is the first member whose prefix exceeds t = u Z; both are
// first worked out in FP32 (weights by bit conversion, scaled by 2^shift each
// side), whose relative error against the FP64 definition is below
//   2^-21 (two truncated squares) + 2^-23 (their sum) + (5 + NCH + 4) 2^-24 < 2^-19
// of the group's sum.  If no member's prefix is within 2^-17 Z of t, every
// comparison has the sign it has in FP64 and the answer is the same; otherwise
// (about one draw in 2^16 / members), or if the sum left the float range,
// the FP64 scans decide.  With FP64 scans alone, bound by the FP64 pipe, the
// kernel took 175 us for 65,536 groups of 64.
template <int NCH>
__global__ void __launch_bounds__(256) k_sample_narrow(SampleParams p, int batch) {
  report_word(p.rep, p.plan_status);
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int l = 1 << p.h;
  const uint2 key = make_uint2((uint32_t)p.seed, (uint32_t)(p.seed >> 32));
  const int shift = p.n_qubits >> 1;           // amplitudes near 2^(-n/2)
  // a warp draws `batch` (at most 32) consecutive samples, lane b their random numbers
  const int64_t i0 = warp * batch;
  if (i0 >= p.n) return;
  const int64_t mine = i0 + (lane < batch ? lane : 0);
  const uint4 r = philox4x32_10(make_uint4((uint32_t)mine, (uint32_t)((uint64_t)mine >> 32), 0u, 0u), key);
  const bool mixed = p.mix > 0.0 && u53(r.x, r.y) < p.mix;
  const unsigned mixed_lanes = __ballot_sync(0xffffffffu, mixed);
  const double u_mine = u53(r.z, r.w);
  const int m = (int)min((int64_t)batch, p.n - i0);
#pragma unroll 2
  for (int b = 0; b < m; ++b) {
    const int64_t i = i0 + b;
    if ((mixed_lanes >> b) & 1) {
      if (lane == 0) p.out[i] = uniform_string(p, i, key);
      continue;
    }
    const int64_t g = i % p.L;
    const double2* __restrict__ Hg = p.H + (g << p.h);
    const double u_pick = __shfl_sync(0xffffffffu, u_mine, b);
    float s[NCH], carry = 0.0f;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      s[c] = 0.0f;
      if (c * 32 + lane < l) {
        const double2 v = __ldg(Hg + c * 32 + lane);
        const float x = abs_as_float(v.x, shift), y = abs_as_float(v.y, shift);
        s[c] = fmaf(x, x, y * y);
      }
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
#pragma unroll
      for (int c = 0; c < NCH; ++c) {
        const float u = __shfl_up_sync(0xffffffffu, s[c], d);
        if (lane >= d) s[c] += u;
      }
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
      s[c] += carry;
      carry = __shfl_sync(0xffffffffu, s[c], 31);
    }
    const float t = (float)u_pick * carry, tol = 0x1.0p-17f * carry;
    int64_t mu = -1;
    bool sure = carry > 0x1.0p-60f && carry < 0x1.0p60f;
#pragma unroll
    for (int c = NCH - 1; c >= 0; --c) {
      const float d = s[c] - t;
      const bool in = c * 32 + lane < l;
      sure = sure && !(in && !(fabsf(d) > tol));
      const unsigned ball = __ballot_sync(0xffffffffu, in && d > 0.0f);
      if (ball) mu = c * 32 + __ffs(ball) - 1;
    }
    if (!__all_sync(0xffffffffu, sure) || mu < 0) mu = scan_total_and_pick(Hg, l, u_pick);
    const uint64_t out = bitstring_of(p, g, mu);
    if (lane == 0) p.out[i] = out;
  }
}

// Methods 1 and 2, a thread per sample (each is a serial chain of its own):
//   1: Metropolis chain with uniform proposals (the paper's in-group MCMC,
//      Method and Supplement): start at member 0; for t < T, propose
//      mu' = bits of Philox(i, 2, t), accept when u * w(mu) < w(mu');
//   2: frugal rejection sampling (Supplement, bitstring choice): for t < 64 M
//      rounds, draw mu = bits of Philox(i, 3, t) and accept when
//      (u * M) * Z < w(mu) * l; after the last round keep mu.  Z is the last
//      of the group's prefix sums.
__global__ void __launch_bounds__(128) k_sample_chain(SampleParams p) {
  report_word(p.rep, p.plan_status);
  const int64_t l = 1LL << p.h, nch = (l + 31) >> 5;
  const uint2 key = make_uint2((uint32_t)p.seed, (uint32_t)(p.seed >> 32));
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < p.m; j += (int64_t)gridDim.x * blockDim.x) {
    int64_t g;
    const int64_t i = sample_of(p, j, g);
    const uint32_t ilo = (uint32_t)i, ihi = (uint32_t)((uint64_t)i >> 32);
    if (p.mix > 0.0) {
      const uint4 r = philox4x32_10(make_uint4(ilo, ihi, 0u, 0u), key);
      if (u53(r.x, r.y) < p.mix) {
        p.out[i] = uniform_string(p, i, key);
        continue;
      }
    }
    const double2* __restrict__ Hg = p.H + (g << p.h);
    int64_t mu = 0;
    if (p.method == 1) {
      double wc = weight_rn(Hg[0]);
      for (int64_t t = 0; t < p.param; ++t) {
        const uint4 q = philox4x32_10(make_uint4(ilo, ihi, 2u, (uint32_t)t), key);
        const int64_t prop = (int64_t)(q.x & (uint32_t)(l - 1));
        const double wp = weight_rn(Hg[prop]);
        const double u = u53(q.z, q.w);
        if (__dmul_rn(u, wc) < wp) { mu = prop; wc = wp; }
      }
    } else {
      const double Z = p.carry[(g - p.g0) * (nch + 1) + nch];
      const double bound = __dmul_rn((double)p.param, Z);
      for (int64_t t = 0; t < 64 * p.param; ++t) {
        const uint4 q = philox4x32_10(make_uint4(ilo, ihi, 3u, (uint32_t)t), key);
        mu = (int64_t)(q.x & (uint32_t)(l - 1));
        const double u = u53(q.z, q.w);
        if (__dmul_rn(u, bound) < __dmul_rn(weight_rn(Hg[mu]), (double)l)) break;
      }
    }
    uint64_t s = p.tails[g] & ~p.open_mask;
    for (int j = 0; j < p.h; ++j) s |= (uint64_t)((mu >> j) & 1) << p.open_q[j];
    p.out[i] = s;
  }
}

// Exact draws read a narrow group once per sample; with more than a few samples
// a group, or from 256 members up, its prefix sums are worked out first.
static bool exact_by_prefix(int64_t L, int h, int64_t n) { return h >= 8 || (h >= 6 && n > 4 * L); }

size_t sample_scratch_doubles(int h, int64_t groups) { return (size_t)(groups * ((((1LL << h) + 31) >> 5) + 1)); }

int64_t sample_groups(int64_t L, int h, int64_t n, int method, size_t max_bytes) {
  if (method == 1 || (method == 0 && !exact_by_prefix(L, h, n))) return 0;
  const int64_t fit = (int64_t)std::min<size_t>(max_bytes / 8 / sample_scratch_doubles(h, 1), (size_t)1 << 62);
  return std::max<int64_t>(1, std::min(std::min(L, n), fit));
}

static cudaError_t launch_sample_window(const SampleParams& p, cudaStream_t s);

// Samples from wide groups need the prefix sums of their groups, 1/64 of the
// head's size for groups from 32 members up.  Where the caller has scratch for
// fewer groups, they are taken in windows, one after another in the same scratch.
cudaError_t launch_sample(const SampleParams& q, cudaStream_t s) {
  if (q.n <= 0) return cudaSuccess;
  SampleParams p = q;
  p.g0 = p.win = 0;
  p.m = p.n;
  const int64_t ng = sample_groups(p.L, p.h, p.n, p.method);   // groups drawn from, or 0: no scratch
  if (ng == 0) return launch_sample_window(p, s);
  if (!p.carry || p.carry_groups < 1) return cudaErrorInvalidValue;
  for (int64_t g0 = 0; g0 < ng; g0 += p.carry_groups) {
    const int64_t w = std::min(p.carry_groups, ng - g0);
    const double2* first = p.H + (g0 << p.h);
    k_group_prefix<<<(unsigned)std::min<int64_t>(w, (int64_t)kSMs * 8), 256, 0, s>>>(first, p.h, w, p.carry);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (w < ng) {
      p.g0 = g0;
      p.win = w;
      p.m = p.n / p.L * w + std::max<int64_t>(0, std::min(p.n % p.L - g0, w));
    }
    e = launch_sample_window(p, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

static cudaError_t launch_sample_window(const SampleParams& p, cudaStream_t s) {
  if (p.method != 0) {
    const int64_t grid = std::min<int64_t>((p.m + 127) / 128, (int64_t)kSMs * 16);
    k_sample_chain<<<(unsigned)grid, 128, 0, s>>>(p);
  } else if (exact_by_prefix(p.L, p.h, p.n)) {
    const int64_t grid = std::min<int64_t>((p.m * 32 + 255) / 256, (int64_t)kSMs * 16);
    k_sample_prefix<<<(unsigned)grid, 256, 0, s>>>(p);
  } else {
    // consecutive samples per warp once there are more samples than warps
    // on the chip: their random numbers cost one Philox evaluation per lane
    const int batch = (int)std::max<int64_t>(1, std::min<int64_t>(32, p.n / (kSMs * 48)));
    const int64_t blocks = ((p.n + batch - 1) / batch + 7) / 8;
    if (p.h <= 5) k_sample_narrow<1><<<(unsigned)blocks, 256, 0, s>>>(p, batch);
    else if (p.h == 6) k_sample_narrow<2><<<(unsigned)blocks, 256, 0, s>>>(p, batch);
    else k_sample_narrow<4><<<(unsigned)blocks, 256, 0, s>>>(p, batch);
  }
  return cudaGetLastError();
}

}  // namespace tn
