// Direct contraction step: C[p][c][r] = sum_k X[mapX(p)][r,k] Y[mapY(p)][k,c] in
// complex64 on the CUDA cores, reading both operands where they lie (any leg
// order), with no permuted or prepared copy of either.
//
// What it is for.  A GEMM step on the tensor cores is three dependent launches
// (permute of A, preparation of B, the GEMM), each of which costs microseconds
// however small the step is, and its 128-row tiles do full work for one useful
// row.  Two kinds of step gain from one launch of plain FP32 arithmetic:
//   - small ones, bound by launches and latency;
//   - narrow ones with a long K (a few rows and columns per pattern), bound by
//     reading the big operand once: the three-launch form writes and reads its
//     split copy on top.
// The planner compares the two forms' modelled times (layout_steps, tc_seconds).
//
// Measured (CUDA events around each launch, of which about 4 us are the
// events'; three launches, then one of this kernel):
//   rows x columns x K            patterns   three launches   direct
//   2^8  x 2^6  x 2^2                    1        23 us          7 us   latency
//   2^12 x 2^8  x 2^4                    1        26 us         10 us   latency
//   2^15 x 2^8  x 2^4                    1        50 us         35 us   FP32, stores
//   2^7  x 2^2  x 2^11                 128       182 us         84 us   FP32
//   2^4  x 2^2  x 2^15                1024     14.44 ms       1.07 ms   HBM, 5.0 TB/s
//   2^18 x 1 x 2^6, X shared            53      2.48 ms       0.19 ms   FP32 (folded)
//   2^12 x 2^12 x 2^8                    1       186 us        688 us   FP32: stays a GEMM
//
// Layout.  X and Y are arrays over binary legs; a CTA's tile covers TR rows
// (the lowest row legs), TC columns and TK values of k per pipeline stage.
// The elements of a stage are enumerated in the order of their addresses (the
// tile's legs sorted by their position in the operand), so that consecutive
// threads read consecutive addresses as far as the tile's legs allow, and are
// copied to Xs[k][row] and Ys[k][col] by 8-byte cp.async.  Every tile element
// is a fixed bit scatter of its index, which a thread works out once: the
// offsets stay in registers for all stages, and there are no tables to load.
//
// Work split.  256 threads form (row groups) x (column groups) x KG groups of k:
// a wide tile has KG = 1, a narrow one splits each stage's k over up to 64
// groups, whose partial sums are added in group order through shared memory.
// When a launch has fewer tiles than the chip has room for and K is long, a
// cluster of up to 8 CTAs splits K further; the partial tiles are added in
// rank order through distributed shared memory.  Every order is fixed, so the
// same inputs give the same bits.
//
// BF16x3 plans.  A step of such a plan that would run in bf16 keeps that
// engine's arithmetic here: the three products of bf16 parts, in FP32.  With
// plain FP32 products in some steps the amplitudes move by as much as the
// engine's own error (2e-5).
//
// Folded patterns.  When all patterns share X, the columns run over (pattern,
// column): one tile serves several patterns and X is read once for all of them.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "batch.cuh"
#include "direct.h"
#include "kernels.h"

namespace tn {

namespace {

__device__ __forceinline__ void cp8(float2* dst, const float2* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ uint32_t cluster_rank_of() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float2 ld_peer(const float2* local, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(a)
               : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}

__device__ __forceinline__ void cmul_acc(float2& acc, float2 a, float2 b) {
  acc.x = fmaf(a.x, b.x, acc.x);
  acc.x = fmaf(-a.y, b.y, acc.x);
  acc.y = fmaf(a.x, b.y, acc.y);
  acc.y = fmaf(a.y, b.x, acc.y);
}

// Offset of index v scattered to the bit positions pos[0..n): bit j of v
// goes to position pos[j].  Lane j works out bit j, one warp-wide OR joins them.
__device__ __forceinline__ uint32_t scatter_warp(uint32_t v, const uint8_t* pos, int n) {
  const int lane = threadIdx.x & 31;
  const uint32_t b = lane < n ? ((v >> lane) & 1u) << pos[lane] : 0u;
  return __reduce_or_sync(0xffffffffu, b);
}

}  // namespace

constexpr int kDirectStages = 3;

template <int TRB, int TCB, int RM, int RN, int TKB>
struct DirectTile {
  static constexpr int TR = 1 << TRB, TC = 1 << TCB, TK = 1 << TKB;
  static constexpr int NRG = TR / RM, NCG = TC / RN, KG = 256 / (NRG * NCG);
  static constexpr int LDX = direct_ldx(TRB), LDY = direct_ldy(TCB);
  static constexpr int STAGE = TK * (LDX + LDY) + (TK * LDY & 1);   // float2 per stage, even
  static constexpr int RED = (KG > 1 ? KG + 1 : 1) * TR * TC;        // float2 of the reductions
  static constexpr int SMEM = 8 * (kDirectStages * STAGE > RED ? kDirectStages * STAGE : RED);
  static constexpr int NX = TR * TK / 256, NY = TC * TK >= 256 ? TC * TK / 256 : 1;
  static_assert(RM % 2 == 0 && NX >= 1 && KG >= 1 && KG <= TK, "tile");
};

// x as a bf16 (rounded to nearest even) and the bf16 of the remainder
__device__ __forceinline__ void split_bf16(float2 x, float2& hi, float2& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x.x, x.y);
  hi = __bfloat1622float2(h);
  lo = __bfloat1622float2(__floats2bfloat162_rn(x.x - hi.x, x.y - hi.y));
}

template <int TRB, int TCB, int RM, int RN, int TKB, bool BF16>
__global__ void __launch_bounds__(256) k_direct(const __grid_constant__ DirectParams p) {
  using T = DirectTile<TRB, TCB, RM, RN, TKB>;
  constexpr int TR = T::TR, TC = T::TC, KG = T::KG, LDX = T::LDX, LDY = T::LDY, NX = T::NX, NY = T::NY;
  extern __shared__ __align__(16) float2 sm[];
  __shared__ unsigned int s_amax;
  const int tid = threadIdx.x, lane = tid & 31;
  const int CL = p.cluster;
  const uint32_t rank = CL > 1 ? cluster_rank_of() : 0u;
  if (tid == 0) s_amax = 0u;

  // tile coordinates: column tiles vary fastest, then row tiles, then patterns
  uint32_t t = CL > 1 ? blockIdx.x / (uint32_t)CL : blockIdx.x;
  const uint32_t rp = p.col_tiles == 1 ? t : t / p.col_tiles;
  const uint32_t ct = t - rp * p.col_tiles;
  const uint32_t rt = rp & ((1u << p.n_rrest) - 1);
  const int64_t pc = rp >> p.n_rrest;

  const int trb = min(p.nr, TRB), tkb = min(p.nk, TKB), tcb = min(p.nc, TCB);
  const int nx = 1 << (trb + tkb);
  const int ny = 1 << (p.fold ? TCB + tkb : tcb + tkb);   // folded: the tile's columns span patterns
  const int over = p.nc - TCB;                            // folded: log2 of the tiles per pattern, or below 0
  const int64_t pc0 = !p.fold ? pc : over >= 0 ? (int64_t)(ct >> over) : (int64_t)ct << -over;
  const uint32_t ctl = !p.fold ? ct : over > 0 ? ct & ((1u << over) - 1) : 0u;

  auto map_of = [](int mode, const uint32_t* tab, int64_t q) {
    return mode == 0 ? q : (mode == 1 ? (int64_t)0 : (int64_t)__ldg(tab + q));
  };
  const int bz = blockIdx.y;
  const float2* Xp = p.X + batch_offset(p, p.bA, bz) + (p.fold ? 0 : map_of(p.mapX_mode, p.mapX, pc) * p.x_pstride) +
                     scatter_warp(rt, p.rrest, p.n_rrest);
  const uint32_t ybase = scatter_warp(ctl, p.crest, p.n_crest);

  // this thread's elements of a stage, tid + 256 e: source offset and shared-
  // memory slot are sums over the bits of the index (of tid once, of e on top)
  uint32_t xo = 0, xs = 0, yo = 0, ys = 0;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const uint32_t bit = (tid >> b) & 1;
    xo += bit * p.xoff[b];
    xs += bit * p.xslot[b];
    yo += bit * p.yoff[b];
    ys += bit * p.yslot[b];
  }
  uint32_t xoe[NX], xse[NX];
#pragma unroll
  for (int e = 0; e < NX; ++e) {
    xoe[e] = xo;
    xse[e] = xs;
#pragma unroll
    for (int b = 0; (1 << b) < NX; ++b)
      if ((e >> b) & 1) {
        xoe[e] += p.xoff[8 + b];
        xse[e] += p.xslot[8 + b];
      }
  }
  const float2* yp[NY];
  const float2* Yb = p.Y + batch_offset(p, p.bB, bz);
  uint32_t yse[NY];
#pragma unroll
  for (int e = 0; e < NY; ++e) {
    uint32_t o = yo, u = ys;
#pragma unroll
    for (int b = 0; (1 << b) < NY; ++b)
      if ((e >> b) & 1) {
        o += p.yoff[8 + b];
        u += p.yslot[8 + b];
      }
    int64_t q = pc0;
    if (p.fold) q = min(pc0 + ((tid + 256 * e) >> (tcb + tkb)), p.PC - 1);   // past the last pattern: read, never stored
    yp[e] = Yb + map_of(p.mapY_mode, p.mapY, q) * p.y_pstride + ybase + o;
    yse[e] = u;
  }

  const int nch = 1 << (p.nk - tkb);                     // stages of the whole K
  const int my = (nch - (int)rank + CL - 1) / CL;        // stages of this CTA: rank, rank + CL, ...
  auto issue = [&](int j, int buf) {
    if (j < my) {
      const uint32_t c = rank + (uint32_t)j * CL;
      const uint32_t hx = scatter_warp(c, p.kxrest, p.nk - tkb), hy = scatter_warp(c, p.kyrest, p.nk - tkb);
      float2* xb = sm + buf * T::STAGE;
      float2* yb = xb + T::TK * LDX;
#pragma unroll
      for (int e = 0; e < NX; ++e)
        if (tid + 256 * e < nx) cp8(xb + xse[e], Xp + xoe[e] + hx);
#pragma unroll
      for (int e = 0; e < NY; ++e)
        if (tid + 256 * e < ny) cp8(yb + yse[e], yp[e] + hy);
    }
    cp_commit();                                          // an empty group past the end keeps the count uniform
  };

  const int rg = tid % T::NRG, cg = (tid / T::NRG) % T::NCG, kg = tid / (T::NRG * T::NCG);
  float2 acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = make_float2(0.f, 0.f);

#pragma unroll
  for (int s = 0; s < kDirectStages - 1; ++s) issue(s, s);
  int buf = 0;
  const int tk = 1 << tkb;
  for (int j = 0; j < my; ++j) {
    cp_wait<kDirectStages - 2>();
    __syncthreads();                                      // stage j is in; the buffer read last round is free
    issue(j + kDirectStages - 1, (buf + kDirectStages - 1) % kDirectStages);
    const float2* xb = sm + buf * T::STAGE;
    const float2* yb = xb + T::TK * LDX;
    buf = (buf + 1) % kDirectStages;
#pragma unroll 4
    for (int k = kg; k < tk; k += KG) {
      float2 a[RM], b[RN];
#pragma unroll
      for (int i = 0; i < RM; i += 2) {
        const float4 v = *(const float4*)(xb + k * LDX + (i / 2) * (2 * T::NRG) + 2 * rg);
        a[i] = make_float2(v.x, v.y);
        a[i + 1] = make_float2(v.z, v.w);
      }
      if constexpr (RN % 2 == 0) {
#pragma unroll
        for (int c = 0; c < RN; c += 2) {
          const float4 v = *(const float4*)(yb + k * LDY + cg * RN + c);
          b[c] = make_float2(v.x, v.y);
          b[c + 1] = make_float2(v.z, v.w);
        }
      } else {
        b[0] = yb[k * LDY + cg];
      }
      if constexpr (BF16) {
        // the BF16x3 products, correction terms first
        float2 al[RM], bl[RN];
#pragma unroll
        for (int i = 0; i < RM; ++i) split_bf16(a[i], a[i], al[i]);
#pragma unroll
        for (int c = 0; c < RN; ++c) split_bf16(b[c], b[c], bl[c]);
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
          for (int c = 0; c < RN; ++c) {
            cmul_acc(acc[i][c], a[i], bl[c]);
            cmul_acc(acc[i][c], al[i], b[c]);
            cmul_acc(acc[i][c], a[i], b[c]);
          }
      } else {
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
          for (int c = 0; c < RN; ++c) cmul_acc(acc[i][c], a[i], b[c]);
      }
    }
  }
  cp_wait<0>();

  // C[pattern][column][row], rows lowest; with folded patterns the column
  // index runs on across patterns, which is the same address
  const int64_t rows = 1LL << p.nr;
  float2* Cp = p.C + batch_offset(p, p.bC, bz) + (p.fold ? 0 : pc * p.c_pstride);
  const int64_t row0 = (int64_t)rt << TRB, col0 = (int64_t)ct << TCB;
  float tmax = 0.0f;
  if (KG == 1 && CL == 1) {
#pragma unroll
    for (int c = 0; c < RN; ++c) {
      const int64_t col = col0 + cg * RN + c;
      if (col >= p.cols) continue;
#pragma unroll
      for (int i = 0; i < RM; i += 2) {
        const int64_t row = row0 + (i / 2) * (2 * T::NRG) + 2 * rg;
        if (row >= rows) continue;
        float2* dst = Cp + (col << p.nr) + row;
        const float2 u = acc[i][c], w = acc[i + 1][c];
        tmax = fmaxf(tmax, fmaxf(fabsf(u.x), fabsf(u.y)));
        if (row + 1 < rows) {
          tmax = fmaxf(tmax, fmaxf(fabsf(w.x), fabsf(w.y)));
          if (p.vec) {
            *(float4*)dst = make_float4(u.x, u.y, w.x, w.y);
          } else {
            dst[0] = u;
            dst[1] = w;
          }
        } else {
          dst[0] = u;
        }
      }
    }
  } else {
    __syncthreads();                                      // every stage buffer is free
    float2* part = sm + (KG > 1 ? TR * TC : 0);           // [KG][TC][TR], this CTA's sum in sm[0..TR*TC)
#pragma unroll
    for (int c = 0; c < RN; ++c)
#pragma unroll
      for (int i = 0; i < RM; ++i)
        part[(kg * TC + cg * RN + c) * TR + (i >> 1) * (2 * T::NRG) + 2 * rg + (i & 1)] = acc[i][c];
    __syncthreads();
    if (KG > 1) {
      for (int o = tid; o < TR * TC; o += 256) {
        float2 s = part[o];
#pragma unroll 8
        for (int g = 1; g < KG; ++g) {
          const float2 v = part[g * TR * TC + o];
          s.x += v.x;
          s.y += v.y;
        }
        sm[o] = s;
      }
    }
    if (CL > 1) cluster_sync(); else __syncthreads();
    for (int o = tid + 256 * (int)rank; o < TR * TC; o += 256 * CL) {
      const int64_t row = row0 + (o & (TR - 1)), col = col0 + (o >> TRB);
      if (row >= rows || col >= p.cols) continue;
      float2 s = CL > 1 ? ld_peer(sm + o, 0) : sm[o];
      for (int r = 1; r < CL; ++r) {
        const float2 v = ld_peer(sm + o, (uint32_t)r);
        s.x += v.x;
        s.y += v.y;
      }
      Cp[(col << p.nr) + row] = s;
      tmax = fmaxf(tmax, fmaxf(fabsf(s.x), fabsf(s.y)));
    }
    if (CL > 1) cluster_sync();                           // peers may still read this CTA's sum
  }
  if (p.amax) {
    const unsigned int m = __reduce_max_sync(0xffffffffu, __float_as_uint(tmax));
    __syncthreads();
    if (lane == 0) atomicMax(&s_amax, m);
    __syncthreads();
    if (tid == 0 && s_amax) atomicMax(p.amax + bz * p.amax_stride, s_amax);
  }
}

namespace {

typedef void (*DirectKernel)(DirectParams);
struct DirectEntry {
  DirectKernel fn[2];      // FP32 products, BF16x3 products
  int smem;
};
#define DIRECT_ENTRY(a, b, c, d, e) \
  {{k_direct<a, b, c, d, e, false>, k_direct<a, b, c, d, e, true>}, DirectTile<a, b, c, d, e>::SMEM}
// in the order of kDirectConfigs (direct.h)
const DirectEntry kEntries[kNumDirectConfigs] = {
    DIRECT_ENTRY(6, 6, 4, 4, 4), DIRECT_ENTRY(6, 5, 4, 4, 4), DIRECT_ENTRY(6, 4, 4, 4, 5), DIRECT_ENTRY(6, 2, 4, 4, 5),
    DIRECT_ENTRY(6, 0, 4, 1, 5),
    DIRECT_ENTRY(4, 4, 4, 4, 6), DIRECT_ENTRY(4, 2, 4, 4, 7), DIRECT_ENTRY(4, 0, 4, 1, 7),
};

}  // namespace

cudaError_t prepare_direct() {
  for (const DirectEntry& e : kEntries) {
    for (DirectKernel fn : e.fn) {
      const cudaError_t r = cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, e.smem);
      if (r != cudaSuccess) return r;
    }
  }
  return cudaSuccess;
}

cudaError_t launch_direct(const DirectParams& p, int config, cudaStream_t s, bool prepare) {
  if (config < 0 || config >= kNumDirectConfigs) return cudaErrorInvalidValue;
  const int64_t tiles = ((int64_t)p.col_tiles << p.n_rrest) * (p.fold ? 1 : p.PC);
  if (tiles < 1 || tiles * p.cluster > 0x7fffffffLL) return cudaErrorInvalidValue;
  const DirectEntry& e = kEntries[config];
  if (prepare) {
    const cudaError_t r =
        cudaFuncSetAttribute((const void*)e.fn[p.bf16 != 0], cudaFuncAttributeMaxDynamicSharedMemorySize, e.smem);
    if (r != cudaSuccess) return r;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * p.cluster), (unsigned)p.n_batch);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = (size_t)e.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)p.cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = p.cluster > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, e.fn[p.bf16 != 0], p);
}

}  // namespace tn
