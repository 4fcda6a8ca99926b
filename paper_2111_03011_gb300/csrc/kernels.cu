// Streaming kernels of the contraction path (HBM-bound steps), the plain
// FP32 CUDA-core complex GEMM and slice accumulation.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstdio>

#include "batch.cuh"
#include "kernels.h"

namespace tn {

static constexpr int kSMs = 152;

__device__ __forceinline__ int64_t map_p(int mode, const uint32_t* tab, int64_t p) {
  return mode == 0 ? p : (mode == 1 ? 0 : (int64_t)__ldg(tab + p));
}

__device__ __forceinline__ float2 cmul_add(float2 acc, float2 a, float2 b) {
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.x = fmaf(-a.y, b.y, acc.x);
  acc.y = fmaf(a.x, b.y, acc.y);
  acc.y = fmaf(a.y, b.x, acc.y);
  return acc;
}

// ------------------------------------------------------------------ K8 / K3
// Small-operand contraction (a gate-like tensor of <= 16x16 applied to a big
// one).  Each thread owns one row m of the big operand: it gathers the 2^NK
// elements addressed by the contracted legs, multiplies by the small operand
// held in shared memory, and writes 2^NN outputs.  Consecutive threads touch
// consecutive addresses, so loads and stores coalesce whatever the leg layout.
template <int NK, int NN>
__global__ void __launch_bounds__(256) k_small(SmallParams p) {
  constexpr int KK = 1 << NK, NNN = 1 << NN;
  __shared__ float2 Bs[KK][NNN];
  int64_t offK[KK];
#pragma unroll
  for (int k = 0; k < KK; ++k) {
    int64_t o = 0;
#pragma unroll
    for (int j = 0; j < NK; ++j)
      if ((k >> j) & 1) o |= 1LL << p.kpos[j];
    offK[k] = o;
  }
  const int bz = blockIdx.z;
  const float2* __restrict__ A0 = p.A + batch_offset(p, p.bA, bz);
  const float2* __restrict__ B0 = p.B + batch_offset(p, p.bB, bz);
  float2* __restrict__ C0 = p.C + batch_offset(p, p.bC, bz);
  const int64_t rowsC = p.M;  // C stride of the n index
  __shared__ unsigned int s_amax;
  if (threadIdx.x == 0) s_amax = 0u;
  float tmax = 0.0f;
  for (int64_t pc = blockIdx.y; pc < p.PC; pc += gridDim.y) {
    const int64_t pa = map_p(p.mapA_mode, p.mapA, pc);
    const int64_t pb = map_p(p.mapB_mode, p.mapB, pc);
    __syncthreads();
    for (int i = threadIdx.x; i < KK * NNN; i += blockDim.x) {
      const int k = i / NNN, n = i % NNN;
      Bs[k][n] = B0[pb * p.b_pstride + p.boffK[k] + p.boffN[n]];
    }
    __syncthreads();
    const float2* __restrict__ Ap = A0 + pa * p.a_pstride;
    float2* __restrict__ Cp = C0 + pc * p.c_pstride;
    for (int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; m < p.M; m += (int64_t)gridDim.x * blockDim.x) {
      int64_t x = m;
#pragma unroll
      for (int j = 0; j < NK; ++j) {
        const int pos = p.kpos[j];
        x = ((x >> pos) << (pos + 1)) | (x & ((1LL << pos) - 1));
      }
      float2 a[KK];
#pragma unroll
      for (int k = 0; k < KK; ++k) a[k] = __ldg(Ap + x + offK[k]);
#pragma unroll
      for (int n = 0; n < NNN; ++n) {
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < KK; ++k) acc = cmul_add(acc, a[k], Bs[k][n]);
        Cp[m + (int64_t)n * rowsC] = acc;
        tmax = fmaxf(tmax, fmaxf(fabsf(acc.x), fabsf(acc.y)));
      }
    }
  }
  if (p.amax) {
    // block maximum of the output (FP16x3 scale of the next GEMM operand)
    unsigned int b = __reduce_max_sync(0xffffffffu, __float_as_uint(tmax));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) atomicMax(&s_amax, b);
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(p.amax + bz * p.amax_stride, s_amax);
  }
}

template <int NK, int NN>
static cudaError_t launch_small_t(const SmallParams& p, cudaStream_t s) {
  const int threads = 256;
  int64_t bx = (p.M + threads - 1) / threads;
  const int64_t cap = (int64_t)kSMs * 8;
  int64_t by = p.PC < 65535 ? p.PC : 65535;
  if (bx * by > cap * 4) bx = std::max<int64_t>(1, (cap * 4) / by);
  if (bx < 1) bx = 1;
  k_small<NK, NN><<<dim3((unsigned)bx, (unsigned)by, (unsigned)p.n_batch), threads, 0, s>>>(p);
  return cudaGetLastError();
}

typedef cudaError_t (*small_fn)(const SmallParams&, cudaStream_t);
#define SMALL_ROW(NK) {launch_small_t<NK, 0>, launch_small_t<NK, 1>, launch_small_t<NK, 2>, launch_small_t<NK, 3>, launch_small_t<NK, 4>}
static const small_fn small_table[5][5] = {SMALL_ROW(0), SMALL_ROW(1), SMALL_ROW(2), SMALL_ROW(3), SMALL_ROW(4)};

cudaError_t launch_small(const SmallParams& p, cudaStream_t s) {
  if (p.nk < 0 || p.nk > 4 || p.nn < 0 || p.nn > 4) return cudaErrorInvalidValue;
  return small_table[p.nk][p.nn](p, s);
}

// ---------------------------------------------------------------------- K1
// Bit-permutation transpose.  A tile covers the input's low bits and the
// preimages of the output's low bits (grown to 10 bits with further input
// bits); it is read with the input's contiguous order and written with the
// output's, through shared memory.  The tile is padded by one element per 32 so
// that the strided reads of the write phase fall into different banks.
// Every index table is OR-linear in the tile index (a bit goes to a position),
// and the padding is additive over disjoint bits, so a thread keeps the entries
// of its own index in registers and adds those of 256, 512 and 768, which are
// the same for all threads: no table is read per element, and the shared memory
// holds tiles only, so that eight CTAs fit an SM instead of four.  The
// tile's base addresses (the remaining "rest" bits of the tile index scattered
// to their positions) are a warp-wide OR, lane j placing bit j.
// 2^25 elements, split to bf16 planes: 104-119 us with the tables in shared
// memory, now 82-91 us (5.9-6.6 TB/s); 2^29: 1,857 -> 1,391 us.
// SPLIT 1: the output is written as two fp32 planes, tf32-rounded hi and the
// remainder lo; SPLIT 2: two bf16 planes, bf16 hi and the bf16-rounded
// remainder; SPLIT 3: two fp16 planes of the value times the operand's power-
// of-two scale (fp16_scale_exp of its ABSMAX slot) -- the operand formats of
// the three tensor-core GEMM engines.
__device__ __forceinline__ int pad32(int i) { return i + (i >> 5); }

__device__ __forceinline__ float tf32_rn(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// Asynchronous 8-byte global -> shared copies (cp.async): the loads of the
// next tiles land in shared memory without holding registers.
__device__ __forceinline__ void cp_async8(float2* dst, const float2* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Tile buffers of the permute: while one tile is written out, the next
// kPermBufs - 1 are in flight.
constexpr int kPermBufs = 3;

// float2 per buffer
__host__ __device__ inline int perm_tile_stride(int nt) { return (nt + (nt >> 5) + 3) & ~1; }

// Four consecutive outputs of one plane as one 16-byte store (16-bit formats)
// or two (fp32 pairs); the destination index is a multiple of 4.
__device__ __forceinline__ void store4(float2* dst, float2 a, float2 b, float2 c, float2 d) {
  float4* q = (float4*)dst;
  q[0] = make_float4(a.x, a.y, b.x, b.y);
  q[1] = make_float4(c.x, c.y, d.x, d.y);
}
template <typename H2>
__device__ __forceinline__ void store4(H2* dst, H2 a, H2 b, H2 c, H2 d) {
  *(uint4*)dst = make_uint4(*(const uint32_t*)&a, *(const uint32_t*)&b, *(const uint32_t*)&c, *(const uint32_t*)&d);
}

// Split of two reals into the hi and lo parts of a tensor-core operand format
// (FMT 0: tf32-rounded fp32 hi + fp32 remainder; 1: bf16 hi + bf16 remainder;
// 2: fp16 of the value times the scale sc).
template <int FMT>
struct Pair;
template <>
struct Pair<0> {
  using T = float2;
  static __device__ __forceinline__ void split(float a, float b, float, T& h, T& l) {
    h = make_float2(tf32_rn(a), tf32_rn(b));
    l = make_float2(a - h.x, b - h.y);
  }
};
template <>
struct Pair<1> {
  using T = __nv_bfloat162;
  static __device__ __forceinline__ void split(float a, float b, float, T& h, T& l) {
    h = __floats2bfloat162_rn(a, b);
    const float2 f = __bfloat1622float2(h);
    l = __floats2bfloat162_rn(a - f.x, b - f.y);
  }
};
template <>
struct Pair<2> {
  using T = __half2;
  static __device__ __forceinline__ void split(float a, float b, float sc, T& h, T& l) {
    a *= sc;
    b *= sc;
    h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    l = __floats2half2_rn(a - f.x, b - f.y);
  }
};

// Real embedding of B for C_r = A_r B_r with interleaved complex rows:
// Bt[j][i] (j = 2n + jc output column, i = 2k + ic reduction index) is
// [[re, -im], [im, re]] in (jc, ic); stored K-major as hi and lo planes in the
// GEMM engine's operand format (FMT 0: tf32-rounded fp32 hi + fp32 remainder;
// 1: bf16 hi + bf16 remainder; 2: fp16 of the value times the scale sc).  One
// thread per complex element of B: it writes the element's 2 x 2 block as two
// pairs of adjacent reals (rows 2n and 2n + 1) in each plane; consecutive
// threads take consecutive k, so every row segment is written contiguously.
// Its loads coalesce only when B's K legs are its low bits; otherwise the
// plan prepares B with the permute kernel in an embedding mode (split 4-6),
// which reads through a shared-memory tile.
template <int FMT>
__device__ __forceinline__ void bprep_tc(const BPrepParams& p, int64_t block, int64_t blocks) {
  using T = typename Pair<FMT>::T;
  const int64_t K = 1LL << p.nk, N = 1LL << p.nn;
  const int64_t per = K * N;                  // complex elements per pattern
  const int64_t total = p.PB * per;
  T* hi = (T*)p.out;                          // pairs: [PB][2N][K] pairs of reals
  T* lo = hi + 2 * total;
  const float sc = FMT == 2 ? pow2f(fp16_scale_exp(*p.scale)) : 1.0f;
  // kU elements per thread and round, their loads issued before any store,
  // so that a grid of one block per SM (beside a running GEMM) still keeps
  // enough loads in flight
  constexpr int kU = 4;
  const int64_t stride = blocks * 256;
  for (int64_t e0 = block * 256 + threadIdx.x; e0 < total; e0 += kU * stride) {
    float2 b[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t e = e0 + u * stride;
      if (e < total) {
        const int64_t pb = e / per, r = e - pb * per;
        b[u] = p.B[pb * p.b_pstride + p.bk[r & (K - 1)] + p.bn[r >> p.nk]];
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t e = e0 + u * stride;
      if (e >= total) break;
      const int64_t pb = e / per, r = e - pb * per;
      const int64_t n = r >> p.nk, k = r & (K - 1);
      const int64_t o0 = (pb * 2 * N + 2 * n) * K + k;   // pair (2k, 2k+1) of row 2n
      T h, l;
      Pair<FMT>::split(b[u].x, -b[u].y, sc, h, l);
      hi[o0] = h;
      lo[o0] = l;
      Pair<FMT>::split(b[u].y, b[u].x, sc, h, l);
      hi[o0 + K] = h;                                    // row 2n + 1
      lo[o0 + K] = l;
    }
  }
}

// One element v at output index o (of all patterns), in the form SPLIT.
template <int SPLIT>
__device__ __forceinline__ void perm_store(const PermParams& p, int64_t planes, float2 v, int64_t o, float sc) {
  if constexpr (SPLIT >= 4) {
    // the tensor-core B operand: output index o = k + K n of a pattern
    // becomes the 2 x 2 block [[re, -im], [im, re]] at pairs (2k, 2k+1)
    // of rows 2n and 2n + 1 of the [2N][2K] real embedding
    using PT = Pair<SPLIT - 4>;
    using T = typename PT::T;
    T* hi = (T*)p.out;
    T* lo = hi + 2 * planes;
    const int64_t K = 1LL << p.embed_nk;
    const int64_t e0 = 2 * o - (o & (K - 1));
    T h, l;
    PT::split(v.x, -v.y, sc, h, l);
    hi[e0] = h;
    lo[e0] = l;
    PT::split(v.y, v.x, sc, h, l);
    hi[e0 + K] = h;
    lo[e0 + K] = l;
  } else if constexpr (SPLIT >= 1) {
    using PT = Pair<SPLIT - 1>;
    using T = typename PT::T;
    T* hi = (T*)p.out;
    T h, l;
    PT::split(v.x, v.y, sc, h, l);
    hi[o] = h;
    hi[planes + o] = l;
  } else {
    p.out[o] = v;
  }
}

template <int SPLIT>
__device__ __forceinline__ void permute(const PermParams& p, uint32_t block, uint32_t blocks) {
  extern __shared__ float2 tile[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int nt = 1 << p.t;
  const int tstride = perm_tile_stride(nt);
  const int ne = nt >> 8;                   // elements per thread (0: fewer than 256, one for the first nt threads)
  // this thread's tile index and, uniform, the steps by 256 and 512 (their sum is that by 768)
  uint32_t in0 = 0, out0 = 0, slot0 = 0, in1 = 0, in2 = 0, out1 = 0, out2 = 0, slot1 = 0, slot2 = 0;
  const bool v4 = SPLIT < 4 && p.vec4;
  // four-outputs form: thread g takes outputs 4g .. 4g + 3 of the tile
  const int j0 = v4 ? 4 * tid : tid;
  if (tid < nt) in0 = __ldg(p.tab + tid);
  if (j0 < nt) {
    out0 = __ldg(p.tab + nt + j0);
    slot0 = (uint32_t)pad32((int)__ldg(p.tab + 2 * nt + j0));
  }
  if (p.t > 8) in1 = __ldg(p.tab + 256);
  if (p.t > 9) in2 = __ldg(p.tab + 512);
  if (v4) {
    slot1 = (uint32_t)pad32((int)__ldg(p.tab + 2 * nt + 1));
    slot2 = (uint32_t)pad32((int)__ldg(p.tab + 2 * nt + 2));
  } else {
    if (p.t > 8) {
      out1 = __ldg(p.tab + nt + 256);
      slot1 = (uint32_t)pad32((int)__ldg(p.tab + 2 * nt + 256));
    }
    if (p.t > 9) {
      out2 = __ldg(p.tab + nt + 512);
      slot2 = (uint32_t)pad32((int)__ldg(p.tab + 2 * nt + 512));
    }
  }
  // lane j: where bit j of a tile's index goes in the input and in the output
  uint64_t bit_in = 0, bit_out = 0;
  if (lane < p.n_rest) {
    bit_in = 1ULL << p.rest_in[lane];
    bit_out = 1ULL << p.rest_out[lane];
  }
  const uint64_t nrest_mask = (1ULL << p.n_rest) - 1;
  const uint64_t total_tiles = (uint64_t)p.P << p.n_rest;
  const int64_t planes = p.P * p.pstride;
  const float sc = (SPLIT == 3 || SPLIT == 6) ? pow2f(fp16_scale_exp(*p.scale)) : 1.0f;
  auto scatter = [&](uint32_t b, uint64_t bit) -> uint64_t {
    const uint64_t v = (b >> lane) & 1u ? bit : 0ULL;
    const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)v);
    const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(v >> 32));
    return ((uint64_t)hi << 32) | lo;
  };
  // issue the copies of tile blk into buffer buf (an empty group past the
  // end keeps the group count uniform)
  const uint32_t dst0 = (uint32_t)pad32(tid);
  auto issue = [&](uint64_t blk, int buf) {
    if (blk < total_tiles) {
      const uint64_t pp = blk >> p.n_rest;
      const float2* src = p.in + (pp * p.pstride + scatter((uint32_t)(blk & nrest_mask), bit_in)) + in0;
      float2* dst = tile + buf * tstride + dst0;
      if (ne == 4) {
        cp_async8(dst, src);
        cp_async8(dst + 264, src + in1);
        cp_async8(dst + 528, src + in2);
        cp_async8(dst + 792, src + in1 + in2);
      } else if (ne == 2) {
        cp_async8(dst, src);
        cp_async8(dst + 264, src + in1);
      } else if (tid < nt) {
        cp_async8(dst, src);
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int k = 0; k < kPermBufs - 1; ++k) issue((uint64_t)block + (uint64_t)k * blocks, k);
  int buf = 0;
  for (uint64_t blk = block; blk < total_tiles; blk += blocks) {
    cp_async_wait<kPermBufs - 2>();   // this thread's copies of tile blk are done
    __syncthreads();                  // ... and everyone's; the buffer written out last round is free
    issue(blk + (uint64_t)(kPermBufs - 1) * blocks, (buf + kPermBufs - 1) % kPermBufs);
    const uint64_t pp = blk >> p.n_rest;
    const int64_t o = (int64_t)(pp * p.pstride + scatter((uint32_t)(blk & nrest_mask), bit_out)) + out0;
    const float2* t = tile + buf * tstride + slot0;
    buf = (buf + 1) % kPermBufs;
    if constexpr (SPLIT < 4) {
      if (v4) {
        // output bits 0 and 1 are tile bits 0 and 1: outputs 4g .. 4g + 3 of
        // the tile are consecutive in memory, from a 4-aligned index.  Fewer,
        // wider stores, but each warp's shared-memory reads take other tile
        // bits than in the other form, so which is faster depends on the
        // permutation: a schedule variant of its own, chosen by timing.
        if (j0 < nt) {
          const float2 v[4] = {t[0], t[slot1], t[slot2], t[slot1 + slot2]};
          if constexpr (SPLIT == 0) {
            store4(p.out + o, v[0], v[1], v[2], v[3]);
          } else {
            using PT = Pair<SPLIT - 1>;
            using T = typename PT::T;
            T h[4], l[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) PT::split(v[e].x, v[e].y, sc, h[e], l[e]);
            store4((T*)p.out + o, h[0], h[1], h[2], h[3]);
            store4((T*)p.out + planes + o, l[0], l[1], l[2], l[3]);
          }
        }
        continue;
      }
    }
    if (ne == 4) {
      const float2 a = t[0], b = t[slot1], c = t[slot2], d = t[slot1 + slot2];
      perm_store<SPLIT>(p, planes, a, o, sc);
      perm_store<SPLIT>(p, planes, b, o + out1, sc);
      perm_store<SPLIT>(p, planes, c, o + out2, sc);
      perm_store<SPLIT>(p, planes, d, o + out1 + out2, sc);
    } else if (ne == 2) {
      const float2 a = t[0], b = t[slot1];
      perm_store<SPLIT>(p, planes, a, o, sc);
      perm_store<SPLIT>(p, planes, b, o + out1, sc);
    } else if (tid < nt) {
      perm_store<SPLIT>(p, planes, t[0], o, sc);
    }
  }
  cp_async_wait<0>();
}

template <int SPLIT>
__global__ void __launch_bounds__(256) k_permute(PermParams p) {
  permute<SPLIT>(p, blockIdx.x, gridDim.x);
}

// Both operands of a tensor-core GEMM in one launch: the first CTAs prepare B
// (they are few and start first), the others permute and split A.  The two have
// nothing to wait for in each other, and a small B's gather hides under A's.
template <int FMT>
__global__ void __launch_bounds__(256) k_operands(PermParams a, BPrepParams b, uint32_t blocks_b) {
  if (blockIdx.x < blocks_b) bprep_tc<FMT>(b, blockIdx.x, blocks_b);
  else permute<FMT + 1>(a, blockIdx.x - blocks_b, gridDim.x - blocks_b);
}

// Scale slot of the FP16x3 engine: max over the operand of |re| and |im|.
// Non-negative fp32 values order like their bit patterns, so the block maxima
// are merged with an unsigned atomicMax into the slot (zeroed before the pass).
__global__ void __launch_bounds__(256) k_absmax(AbsmaxParams p) {
  __shared__ float red[8];
  float m = 0.0f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += (int64_t)gridDim.x * blockDim.x) {
    const float2 v = __ldg(p.in + i);
    m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) atomicMax(p.out, __float_as_uint(m));
  }
}

cudaError_t launch_absmax(const AbsmaxParams& p, cudaStream_t s) {
  const int64_t grid = std::max<int64_t>(std::min<int64_t>((p.n + 255) / 256, (int64_t)kSMs * 8), 1);
  k_absmax<<<(unsigned)grid, 256, 0, s>>>(p);
  return cudaGetLastError();
}

static size_t perm_smem(int t) { return sizeof(float2) * (size_t)kPermBufs * perm_tile_stride(1 << t); }

cudaError_t launch_permute(const PermParams& p, cudaStream_t s) {
  if (p.n_rest > 32) return cudaErrorInvalidValue;
  const int64_t blocks = (1LL << p.n_rest) * p.P;
  const int64_t grid = std::min<int64_t>(blocks, (int64_t)kSMs * 8);
  if (p.t < 0 || p.t > 10) return cudaErrorInvalidValue;
  const size_t smem = perm_smem(p.t);
  if (p.split == 1) k_permute<1><<<(unsigned)grid, 256, smem, s>>>(p);
  else if (p.split == 2) k_permute<2><<<(unsigned)grid, 256, smem, s>>>(p);
  else if (p.split == 3) k_permute<3><<<(unsigned)grid, 256, smem, s>>>(p);
  else if (p.split == 4) k_permute<4><<<(unsigned)grid, 256, smem, s>>>(p);
  else if (p.split == 5) k_permute<5><<<(unsigned)grid, 256, smem, s>>>(p);
  else if (p.split == 6) k_permute<6><<<(unsigned)grid, 256, smem, s>>>(p);
  else k_permute<0><<<(unsigned)grid, 256, smem, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_operands(const PermParams& a, const BPrepParams& b, cudaStream_t s) {
  if (a.n_rest > 32 || a.t < 0 || a.t > 10 || a.split != b.h16 + 1) return cudaErrorInvalidValue;
  const int64_t total = b.PB << (b.nk + b.nn);
  const uint32_t blocks_b = (uint32_t)std::max<int64_t>(std::min<int64_t>((total + 1023) / 1024, kSMs * 4), 1);
  const uint32_t blocks_a = (uint32_t)std::min<int64_t>((1LL << a.n_rest) * a.P, (int64_t)kSMs * 8);
  const dim3 grid(blocks_a + blocks_b);
  const size_t smem = perm_smem(a.t);
  if (b.h16 == 2) k_operands<2><<<grid, 256, smem, s>>>(a, b, blocks_b);
  else if (b.h16 == 1) k_operands<1><<<grid, 256, smem, s>>>(a, b, blocks_b);
  else k_operands<0><<<grid, 256, smem, s>>>(a, b, blocks_b);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ B prep
__global__ void k_bprep_c(BPrepParams p) {
  const int64_t K = 1LL << p.nk, N = 1LL << p.nn;
  const int64_t total = p.PB * K * N;
  float2* out = (float2*)p.out;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t pb = e / (K * N), r = e % (K * N);
    const int64_t k = r / N, n = r % N;
    out[e] = p.B[pb * p.b_pstride + p.bk[k] + p.bn[n]];
  }
}

template <int FMT>
__global__ void __launch_bounds__(256) k_bprep_tc(BPrepParams p) {
  bprep_tc<FMT>(p, blockIdx.x, gridDim.x);
}

cudaError_t launch_bprep_c(const BPrepParams& p, cudaStream_t s) {
  const int64_t total = p.PB << (p.nk + p.nn);
  const int64_t grid = std::min<int64_t>((total + 255) / 256, (int64_t)kSMs * 8);
  k_bprep_c<<<(unsigned)std::max<int64_t>(grid, 1), 256, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_bprep_tc(const BPrepParams& p, cudaStream_t s, bool beside_gemm) {
  const int64_t total = p.PB << (p.nk + p.nn);
  // beside a running GEMM (one CTA per SM, most of the registers and shared
  // memory): one 256-thread block per SM, which fits next to it
  const int64_t cap = beside_gemm ? (int64_t)kSMs : (int64_t)kSMs * 16;
  const unsigned grid = (unsigned)std::max<int64_t>(std::min<int64_t>((total + 255) / 256, cap), 1);
  if (p.h16 == 2) k_bprep_tc<2><<<grid, 256, 0, s>>>(p);
  else if (p.h16 == 1) k_bprep_tc<1><<<grid, 256, 0, s>>>(p);
  else k_bprep_tc<0><<<grid, 256, 0, s>>>(p);
  return cudaGetLastError();
}

// --------------------------------------------- operands of a standalone GEMM
// Row-major operands need no gather tables: one launch takes the maxima of both
// (16-byte loads), one splits A as a stream and transposes B's tiles of
// 32 k x 32 n through shared memory, so that it is read along n and its
// embedding written along k, both coalesced.  M = 2^13, N = 2^10, K = 2^11 in
// fp16: two maximum passes, permute kernel and gather kernel took 107 us, these
// two launches about 85 us of a 385 us call (the GEMM itself 277 us).
__global__ void __launch_bounds__(256) k_gemm_max(const float2* __restrict__ A, int64_t nA, int blocks_a,
                                                  const float2* __restrict__ B, int64_t nB, int vec,
                                                  unsigned int* scale) {
  __shared__ unsigned int red[8];
  const bool a = (int)blockIdx.x < blocks_a;
  const float2* __restrict__ p = a ? A : B;
  const int64_t n = a ? nA : nB;
  const int64_t b = a ? blockIdx.x : blockIdx.x - blocks_a, nb = a ? blocks_a : gridDim.x - blocks_a;
  float m = 0.0f;
  int64_t done = 0;
  if (vec) {                                    // two elements per load
    done = n & ~(int64_t)1;
    const float4* q = (const float4*)p;
#pragma unroll 4
    for (int64_t i = b * 256 + threadIdx.x; i < n >> 1; i += nb * 256) {
      const float4 v = __ldg(q + i);
      m = fmaxf(fmaxf(fmaxf(m, fabsf(v.x)), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
    }
  }
  for (int64_t i = done + b * 256 + threadIdx.x; i < n; i += nb * 256) {
    const float2 v = __ldg(p + i);
    m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
  }
  const unsigned int w = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = w;
  __syncthreads();
  if (threadIdx.x < 32) {
    const unsigned int t = __reduce_max_sync(0xffffffffu, threadIdx.x < 8 ? red[threadIdx.x] : 0u);
    if (threadIdx.x == 0) atomicMax(scale + (a ? 0 : 1), t);
  }
}

template <int FMT>
__global__ void __launch_bounds__(256) k_gemm_operands(GemmOperands p, int64_t blocks_b, int vec) {
  using PT = Pair<FMT>;
  using T = typename PT::T;
  if ((int64_t)blockIdx.x >= blocks_b) {
    // A: four consecutive elements per thread and round (the count is a
    // multiple of four for the 16-bit formats, of two for tf32)
    const float sc = FMT == 2 ? pow2f(fp16_scale_exp(p.scale[0])) : 1.0f;
    T* hi = (T*)p.a_planes;
    T* lo = hi + p.nA;
    const int64_t first = ((int64_t)blockIdx.x - blocks_b) * 256 + threadIdx.x;
    const int64_t step = ((int64_t)gridDim.x - blocks_b) * 256;
    const int64_t quads = vec ? p.nA >> 2 : 0;
    for (int64_t i = first; i < quads; i += step) {
      const float4 u = __ldg((const float4*)p.A + 2 * i), v = __ldg((const float4*)p.A + 2 * i + 1);
      T h[4], l[4];
      PT::split(u.x, u.y, sc, h[0], l[0]);
      PT::split(u.z, u.w, sc, h[1], l[1]);
      PT::split(v.x, v.y, sc, h[2], l[2]);
      PT::split(v.z, v.w, sc, h[3], l[3]);
      store4(hi + 4 * i, h[0], h[1], h[2], h[3]);
      if (FMT != 0 || (p.nA & 1) == 0) {
        store4(lo + 4 * i, l[0], l[1], l[2], l[3]);
      } else {
        for (int e = 0; e < 4; ++e) lo[4 * i + e] = l[e];
      }
    }
    for (int64_t i = 4 * quads + first; i < p.nA; i += step) {
      const float2 v = __ldg(p.A + i);
      T h, l;
      PT::split(v.x, v.y, sc, h, l);
      hi[i] = h;
      lo[i] = l;
    }
    return;
  }
  __shared__ float2 tile[32][33];
  const float sc = FMT == 2 ? pow2f(fp16_scale_exp(p.scale[1])) : 1.0f;
  T* hi = (T*)p.b_planes;
  T* lo = hi + 2 * p.PB * p.K * p.N;
  const int64_t tk = (p.K + 31) >> 5, tn = (p.N + 31) >> 5;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (int64_t t = blockIdx.x; t < p.PB * tk * tn; t += blocks_b) {
    const int64_t n0 = (t % tn) * 32, k0 = (t / tn % tk) * 32, pb = t / (tn * tk);
    __syncthreads();
#pragma unroll
    for (int j = y; j < 32; j += 8)
      if (k0 + j < p.K && n0 + x < p.N) tile[j][x] = __ldg(p.B + (pb * p.K + k0 + j) * p.N + n0 + x);
    __syncthreads();
#pragma unroll
    for (int j = y; j < 32; j += 8) {
      const int64_t n = n0 + j, k = k0 + x;
      if (n >= p.N || k >= p.K) continue;
      const float2 v = tile[x][j];
      const int64_t o = (pb * 2 * p.N + 2 * n) * p.K + k;   // pair (2k, 2k + 1) of row 2n
      T h, l;
      PT::split(v.x, -v.y, sc, h, l);
      hi[o] = h;
      lo[o] = l;
      PT::split(v.y, v.x, sc, h, l);
      hi[o + p.K] = h;
      lo[o + p.K] = l;
    }
  }
}

cudaError_t launch_gemm_operands(const GemmOperands& p, cudaStream_t s) {
  const int64_t nB = p.PB * p.K * p.N;
  const int vec = (uintptr_t)p.A % 16 == 0;
  const int64_t cap = (int64_t)kSMs * 8;
  if (p.fmt == 2) {
    const int ba = (int)std::min<int64_t>((p.nA + 1023) / 1024, cap), bb = (int)std::min<int64_t>((nB + 1023) / 1024, cap);
    k_gemm_max<<<(unsigned)(ba + bb), 256, 0, s>>>(p.A, p.nA, ba, p.B, nB, vec && (uintptr_t)p.B % 16 == 0, p.scale);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const int64_t bb = std::min<int64_t>(p.PB * ((p.K + 31) / 32) * ((p.N + 31) / 32), cap);
  const int64_t ba = std::min<int64_t>((p.nA + 1023) / 1024, cap);
  const unsigned grid = (unsigned)(ba + bb);
  if (p.fmt == 2) k_gemm_operands<2><<<grid, 256, 0, s>>>(p, bb, vec);
  else if (p.fmt == 1) k_gemm_operands<1><<<grid, 256, 0, s>>>(p, bb, vec);
  else k_gemm_operands<0><<<grid, 256, 0, s>>>(p, bb, vec);
  return cudaGetLastError();
}

// ------------------------------------------------------------ SIMT GEMM
// Plain FP32 complex GEMM on CUDA cores: 64x64 complex tile, 16-deep k slab,
// 4x4 outputs per thread.  The reference "plain complex64" engine.
__global__ void __launch_bounds__(256) k_gemm_simt(GemmParams p) {
  constexpr int BM = 64, BN = 64, BK = 16;
  __shared__ float2 As[BK][BM + 1];
  __shared__ float2 Bs[BK][BN];
  const int64_t tilesN = (p.N + BN - 1) / BN;
  const int64_t tm = blockIdx.x / tilesN, tn = blockIdx.x % tilesN;
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const float2* __restrict__ Bg0 = (const float2*)p.B;
  for (int64_t pc = blockIdx.y; pc < p.PC; pc += gridDim.y) {
    const int64_t pa = map_p(p.mapA_mode, p.mapA, pc), pb = map_p(p.mapB_mode, p.mapB, pc);
    const float2* __restrict__ Ag = p.A + pa * p.M * p.K;
    const float2* __restrict__ Bg = Bg0 + pb * p.K * p.N;
    float2* __restrict__ Cg = p.C + pc * p.M * p.N;
    float2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
    for (int64_t k0 = 0; k0 < p.K; k0 += BK) {
      __syncthreads();
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int e = tid + 256 * r;
        const int ml = e / BK, kl = e % BK;
        const int64_t m = tm * BM + ml, k = k0 + kl;
        As[kl][ml] = (m < p.M && k < p.K) ? __ldg(Ag + m * p.K + k) : make_float2(0.f, 0.f);
        const int kb = e / BN, nl = e % BN;
        const int64_t n = tn * BN + nl, kk = k0 + kb;
        Bs[kb][nl] = (n < p.N && kk < p.K) ? __ldg(Bg + kk * p.N + n) : make_float2(0.f, 0.f);
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        float2 a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = cmul_add(acc[i][j], a[i], b[j]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t m = tm * BM + ty + 16 * i;
      if (m >= p.M) continue;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t n = tn * BN + tx + 16 * j;
        if (n < p.N) Cg[m * p.N + n] = acc[i][j];
      }
    }
  }
}

cudaError_t launch_gemm_simt(const GemmParams& p, cudaStream_t s) {
  const int64_t tiles = ((p.M + 63) / 64) * ((p.N + 63) / 64);
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  const int64_t gy = std::min<int64_t>(p.PC, 65535);
  k_gemm_simt<<<dim3((unsigned)tiles, (unsigned)gy), 256, 0, s>>>(p);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------- K4
// H[g][mu] += F[pidx[g]][open bits of mu]   (FP64 accumulation of slices)
__global__ void k_accum(AccumParams p) {
  const int64_t total = p.L << p.h;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t g = e >> p.h;
    const int64_t mu = e & ((1LL << p.h) - 1);
    int64_t off = (int64_t)__ldg(p.pidx + g) * p.f_pstride;
    for (int j = 0; j < p.h; ++j)
      if ((mu >> j) & 1) off |= 1LL << p.open_pos[j];
    // the passes of a batch are added one after another, as single launches would
    double2 hv = p.H[e];
#pragma unroll 4
    for (int b = 0; b < p.n_batch; ++b) {
      const float2 v = __ldg(p.F + batch_offset(p, p.bA, b) + off);
      hv.x += (double)v.x;
      hv.y += (double)v.y;
    }
    p.H[e] = hv;
  }
}

cudaError_t launch_accum(const AccumParams& p, cudaStream_t s) {
  const int64_t total = p.L << p.h;
  const int64_t grid = std::min<int64_t>((total + 255) / 256, (int64_t)kSMs * 8);
  k_accum<<<(unsigned)std::max<int64_t>(grid, 1), 256, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace tn
