// spatial_simt.cu — spatial importance (Sec. 3.3.1, Eq. 3 with Eq. 4-5) on
// the CUDA cores, for fp32 inputs (which tensor cores cannot take at the fp32
// score tolerance) and for head widths the tensor-core kernel does not tile.
//
// Q K^T is a register-tiled product: a CTA takes TM consecutive image queries
// of one batch element and 128-key tiles; a warp owns RM queries, a lane four
// keys of each (lane, lane + 32, ...), so that a key row's 16-byte reads are
// 32 different rows (no bytes read twice by a warp) and a query row's are one
// broadcast.  Every dot product keeps four partial sums (columns c mod 4).  Q
// and K come in chunks of 32 columns through a 3-stage ring (cp.async for
// fp32, 16-byte loads through registers for bf16).  After a key tile each lane folds its logits into a running (max, sum
// over all keys, sum over text keys) per query in the log2 domain; the lanes
// are merged by shuffles only when the head's keys end.
//
// Work split: the H x ceil(Nk / 128) (head, key tile) items of a query tile go
// to the CTAs of one thread-block cluster in equal contiguous ranges.  A head
// whose keys lie in one CTA gives its text mass there; one that straddles
// CTAs leaves partial statistics.  At the end every CTA pushes its sum of
// masses and its (at most two) partials per row into rank 0's shared memory,
// and rank 0 merges them in rank order: the head mean of Eq. 3 is a sum in a
// fixed order, with no workspace and no atomics.  The text keys are the first
// L, or those a caller's key mask marks (interleaved text and image keys).
//
// Bound by the FMA pipe and what feeds it: per 4 columns a warp issues 128
// FMAs and 12 shared loads of 24 wavefronts (75 % of the FMA time); ncu counts
// 61 % of the issue slots taken, the rest barriers, register ports and load
// latency with 8 warps per SM.  24 heads x 1024 x 1536 x 128 fp32: 3950 -> 310
// us (31 of 74 TFLOP/s; before, one warp per query read each key row for four
// FMAs per 16-byte load, and heads ran one after the other); 2 heads x 256 x
// 288 x 64: 17 -> 6.7 us.  bf16: 24 heads x 1024 x 1536 x 96 2125 -> 317 us (457 with
// elements loaded one by one), x 40 979 -> 180 (259), 8 x 16 heads x 256 x 333 x 256
// 1378 -> 258 (380), 1 head x 64 x 100 x 256 10.5 -> 10.3 (21.9).  Packed f32x2 FMAs, pairs of columns or of keys,
// were no faster (411 us either way with 8 x 4 lanes to a warp's tile), nor
// were 64 rows per CTA (615-640 us, one CTA per SM).
#include "avits_common.cuh"
#include "avits_internal.h"

namespace avits {
namespace {

constexpr int kTN = 128;                 // keys per tile
constexpr int kRN = kTN / 32;            // keys per lane: lane, lane + 32, ...
constexpr int kDK = 32;                  // columns per stage
constexpr int kLd = kDK + 4;             // row stride (floats): 8 rows, 32 banks
constexpr int kStages = 3;
constexpr int kMaxCluster = 8;           // the portable cluster size

__device__ __forceinline__ float fast_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Running row statistics: x = c_log2 * (q.k); the sums are of 2^(x - m).
struct RowStat {
  float m, la, lt;
};

__device__ __forceinline__ void merge_stat(RowStat& a, float m2, float la2, float lt2) {
  const float mx = fmaxf(a.m, m2);
  if (mx == -INFINITY) {   // no key yet, or NaN sums, which stay
    a.la += la2;
    a.lt += lt2;
    return;
  }
  const float f1 = fast_ex2(a.m - mx), f2 = fast_ex2(m2 - mx);
  a.la = a.la * f1 + la2 * f2;
  a.lt = a.lt * f1 + lt2 * f2;
  a.m = mx;
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Store into the shared memory of the cluster's rank 0 at this CTA's offset.
__device__ __forceinline__ void st_rank0(float* local, float v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(local)), "r"(0));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

struct SimtParams {
  const void* q;
  const void* k;
  int B, H, M, Nk, L, d;
  int64_t q_sb, q_sh, q_sn, k_sb, k_sh, k_sn;
  float c_log2, weight;
  int accumulate;
  float* A;
  float* lse;
  const uint8_t* tmask;
  int tiles, n_kt, items, per, cs;   // query tiles; items and items per CTA of a cluster
};

// How a stage's rows come to shared memory.  Elements: one by one.  Async: fp32 in
// 16-byte asynchronous copies.  Vectors: bf16 in 16-byte loads into registers,
// converted and stored once the products of the stage in hand have been issued.
// The last two need d, the strides and the bases to be multiples of 16 bytes
// (checked on the host).
enum Load { kLoadElements, kLoadAsync, kLoadVectors };

// kRows rows (row r0 + r of `base`, valid below `rows`) of columns c0 ..
// c0 + 31 (below d) into ks as fp32, zero where there is no element.
template <typename T, int kRows, int kThreads, bool kAsync>
__device__ __forceinline__ void load_rows(const T* base, int64_t sn, int r0, int rows, int c0,
                                          int d, float* ks) {
  if constexpr (kAsync) {
#pragma unroll
    for (int u = 0; u < kRows * 8 / kThreads; ++u) {
      const int v = threadIdx.x + u * kThreads, r = v >> 3, c = (v & 7) * 4;
      const bool in = r0 + r < rows && c0 + c < d;
      const T* src = in ? base + (int64_t)(r0 + r) * sn + c0 + c : base;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                       smem_u32(ks + r * kLd + c)),
                   "l"(src), "r"(in ? 16 : 0)
                   : "memory");
    }
  } else {
    constexpr int kN = kRows * kDK / kThreads;   // elements per thread
    constexpr int kBatch = kN < 8 ? kN : 8;
    static_assert(kN % kBatch == 0, "whole batches");
#pragma unroll 1
    for (int u0 = 0; u0 < kN; u0 += kBatch) {
      float w[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int v = threadIdx.x + (u0 + u) * kThreads, r = v >> 5, c = v & 31;
        w[u] = (r0 + r < rows && c0 + c < d) ? load_elem(base + (int64_t)(r0 + r) * sn, c0 + c) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int v = threadIdx.x + (u0 + u) * kThreads;
        ks[(v >> 5) * kLd + (v & 31)] = w[u];
      }
    }
  }
}

// A stage of bf16 (kQ query rows, then kTN key rows) in registers on its way to
// shared memory: 8 columns per vector, four vectors per row.
template <int kQ, int kThreads>
struct StageVectors {
  static constexpr int kN = ((kQ + kTN) * 4 + kThreads - 1) / kThreads;
  uint4 w[kN];
  __device__ __forceinline__ void load(const __nv_bfloat16* q, int64_t q_sn, int q0, int q_rows,
                                       const __nv_bfloat16* k, int64_t k_sn, int k0, int k_rows,
                                       int c0, int d) {
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      const int v = threadIdx.x + u * kThreads, c = c0 + (v & 3) * 8;
      const int r = v >> 2;
      const bool of_q = r < kQ;
      const int row = of_q ? q0 + r : k0 + (r - kQ);
      w[u] = make_uint4(0u, 0u, 0u, 0u);
      if (r < kQ + kTN && row < (of_q ? q_rows : k_rows) && c < d)
        w[u] = *reinterpret_cast<const uint4*>((of_q ? q + (int64_t)row * q_sn : k + (int64_t)row * k_sn) + c);
    }
  }
  __device__ __forceinline__ void store(float* st) const {
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      const int v = threadIdx.x + u * kThreads, r = v >> 2;
      if (r >= kQ + kTN) continue;
      float4* dst = reinterpret_cast<float4*>(st + r * kLd + (v & 3) * 8);
      dst[0] = make_float4(bf16_lo(w[u].x), bf16_hi(w[u].x), bf16_lo(w[u].y), bf16_hi(w[u].y));
      dst[1] = make_float4(bf16_lo(w[u].z), bf16_hi(w[u].z), bf16_lo(w[u].w), bf16_hi(w[u].w));
    }
  }
};

template <int TM>
constexpr size_t simt_smem() {
  return (size_t)kStages * (TM + kTN) * kLd * sizeof(float);
}

template <typename T, int TM, int RM, Load kLoad>
__global__ void __launch_bounds__(32 * (TM / RM), 2)
spatial_simt_kernel(const SimtParams p) {
  constexpr int kThreads = 32 * (TM / RM);
  constexpr int kStageFloats = (TM + kTN) * kLd;
  extern __shared__ __align__(16) float stages[];
  // per rank and row the sum of whole heads' masses, the first and the last
  // partial (m, all, text): a CTA fills its own rank's entry, rank 0 gets all
  __shared__ float gather[kMaxCluster][7][TM];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wrow = warp * RM;          // the warp's first row of the tile
  const bool owner = lane < RM;        // this lane takes row wrow + lane's results
  const int cs = p.cs;
  const int rank = cs > 1 ? (int)cluster_rank() : 0;
  const int cl = (int)blockIdx.x / cs;
  const int b = cl / p.tiles, row0 = (cl - b * p.tiles) * TM;
  const int it_begin = rank * p.per, it_end = min(it_begin + p.per, p.items);
  pdl_wait_then_trigger();
  if (cs > 1) cluster_arrive();   // waited for before anything is pushed

  const T* qb = static_cast<const T*>(p.q) + (int64_t)b * p.q_sb;
  const T* kb = static_cast<const T*>(p.k) + (int64_t)b * p.k_sb;
  const uint8_t* mrow = p.tmask ? p.tmask + (int64_t)b * p.Nk : nullptr;
  const int nch = (p.d + kDK - 1) / kDK;
  const float ln2 = 0.69314718055994530942f;

  // the load side runs two stages ahead; vectors: the registers of a stage are
  // loaded by issue() and stored by deliver()
  StageVectors<TM, kThreads> held;
  float* held_for = nullptr;
  int l_it = it_begin, l_ch = 0, l_stage = 0;
  int l_h = it_begin / p.n_kt, l_kt = it_begin - l_h * p.n_kt;
  auto issue = [&]() {
    if (l_it < it_end) {
      float* st = stages + l_stage * kStageFloats;
      if constexpr (kLoad == kLoadVectors) {
        held.load(qb + (int64_t)l_h * p.q_sh, p.q_sn, row0, p.M, kb + (int64_t)l_h * p.k_sh, p.k_sn,
                  l_kt * kTN, p.Nk, l_ch * kDK, p.d);
        held_for = st;
      } else {
        load_rows<T, TM, kThreads, kLoad == kLoadAsync>(qb + (int64_t)l_h * p.q_sh, p.q_sn, row0, p.M,
                                                        l_ch * kDK, p.d, st);
        load_rows<T, kTN, kThreads, kLoad == kLoadAsync>(kb + (int64_t)l_h * p.k_sh, p.k_sn,
                                                         l_kt * kTN, p.Nk, l_ch * kDK, p.d,
                                                         st + TM * kLd);
      }
      if (++l_ch == nch) {
        l_ch = 0;
        ++l_it;
        if (++l_kt == p.n_kt) { l_kt = 0; ++l_h; }
      }
      l_stage = l_stage == kStages - 1 ? 0 : l_stage + 1;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto deliver = [&]() {
    if constexpr (kLoad == kLoadVectors) {
      if (held_for) held.store(held_for);
      held_for = nullptr;
    }
  };
  issue();
  deliver();
  issue();
  deliver();

  RowStat st[RM];
#pragma unroll
  for (int i = 0; i < RM; ++i) st[i] = RowStat{-INFINITY, 0.f, 0.f};
  float* own = &gather[rank][0][wrow + (owner ? lane : 0)];
  if (owner) {
#pragma unroll
    for (int e = 0; e < 7; ++e) own[e * TM] = 0.f;
  }
  int stage = 0;
  int h = it_begin / p.n_kt, kt = it_begin - h * p.n_kt;
  bool seg_start = true, seg_whole = kt == 0;   // this head's keys from the first on
  for (int it = it_begin; it < it_end; ++it) {
    float acc[RM][kRN][4];
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int j = 0; j < kRN; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
    for (int ch = 0; ch < nch; ++ch) {
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncthreads();   // this stage has landed, the one to refill has been read
      issue();
      const float* qs = stages + stage * kStageFloats + wrow * kLd;
      const float* ks = stages + stage * kStageFloats + (TM + lane) * kLd;
      stage = stage == kStages - 1 ? 0 : stage + 1;
      auto step = [&](int c) {
        float4 qv[RM];
#pragma unroll
        for (int i = 0; i < RM; ++i)
          qv[i] = *reinterpret_cast<const float4*>(qs + i * kLd + c);
#pragma unroll
        for (int j = 0; j < kRN; ++j) {
          const float4 kv = *reinterpret_cast<const float4*>(ks + j * 32 * kLd + c);
#pragma unroll
          for (int i = 0; i < RM; ++i) {
            float* a = acc[i][j];
            a[0] = fmaf(qv[i].x, kv.x, a[0]);
            a[1] = fmaf(qv[i].y, kv.y, a[1]);
            a[2] = fmaf(qv[i].z, kv.z, a[2]);
            a[3] = fmaf(qv[i].w, kv.w, a[3]);
          }
        }
      };
      const int left = p.d - ch * kDK;
      if (left >= kDK) {
#pragma unroll 2
        for (int c = 0; c < kDK; c += 4) step(c);
      } else {
#pragma unroll 1
        for (int c = 0; c < left; c += 4) step(c);
      }
      deliver();
    }
    // fold the tile's logits into the row statistics
    const int key0 = kt * kTN + lane;
    uint32_t text = 0u, valid = 0u;   // bit j: key key0 + 32 j
#pragma unroll
    for (int j = 0; j < kRN; ++j) {
      const int key = key0 + j * 32;
      if (key < p.Nk) {
        valid |= 1u << j;
        if (mrow ? mrow[key] != 0 : key < p.L) text |= 1u << j;
      }
    }
    if (valid) {
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        float x[kRN], mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < kRN; ++j) {
          const float* a = acc[i][j];
          x[j] = ((a[0] + a[1]) + (a[2] + a[3])) * p.c_log2;
          if ((valid >> j) & 1u) mx = fmaxf(mx, x[j]);
        }
        if (mx > st[i].m) {
          const float corr = fast_ex2(st[i].m - mx);
          st[i].la *= corr;
          st[i].lt *= corr;
          st[i].m = mx;
        }
        float sa = 0.f, sx = 0.f;
#pragma unroll
        for (int j = 0; j < kRN; ++j) {
          const float e = ((valid >> j) & 1u) ? fast_ex2(x[j] - st[i].m) : 0.f;
          sa += e;
          sx += ((text >> j) & 1u) ? e : 0.f;
        }
        st[i].la += sa;
        st[i].lt += sx;
      }
    }
    const bool head_end = kt == p.n_kt - 1;
    if (head_end || it == it_end - 1) {
      // merge the lanes; lane i keeps the result of row i
      RowStat r{-INFINITY, 0.f, 0.f};
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        float mw = st[i].m;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mw = fmaxf(mw, __shfl_xor_sync(0xffffffffu, mw, o));
        const float f = st[i].m == -INFINITY ? 0.f : fast_ex2(st[i].m - mw);
        float la = st[i].la * f, lt = st[i].lt * f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          la += __shfl_xor_sync(0xffffffffu, la, o);
          lt += __shfl_xor_sync(0xffffffffu, lt, o);
        }
        if (lane == i) r = RowStat{mw, la, lt};
        st[i] = RowStat{-INFINITY, 0.f, 0.f};
      }
      if (owner) {
        if (seg_whole && head_end) {
          own[0] += r.lt / r.la;
          const int row = row0 + wrow + lane;
          if (p.lse && row < p.M) {
            float* lp = p.lse + (((int64_t)b * p.H + h) * p.M + row) * 2;
            lp[0] = (r.m + __log2f(r.la)) * ln2;
            lp[1] = r.lt > 0.f ? (r.m + __log2f(r.lt)) * ln2 : -INFINITY;
          }
        } else {
          float* w = own + (seg_start ? TM : 4 * TM);
          w[0] = r.m;
          w[TM] = r.la;
          w[2 * TM] = r.lt;
        }
      }
      seg_start = false;
      seg_whole = true;
    }
    if (head_end) { kt = 0; ++h; } else { ++kt; }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");

  // push to rank 0, which merges in rank order
  if (cs > 1) cluster_wait();   // every CTA of the cluster runs
  if (rank != 0 && owner) {
#pragma unroll
    for (int e = 0; e < 7; ++e) st_rank0(own + e * TM, own[e * TM]);
  }
  if (cs > 1) {
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }
  if (rank != 0 || tid >= TM || row0 + tid >= p.M) return;
  const int row = row0 + tid;
  float tot = 0.f;
  RowStat cur{-INFINITY, 0.f, 0.f};
  int cur_h = -1;
  auto flush = [&]() {
    if (cur_h < 0) return;
    tot += cur.lt / cur.la;
    if (p.lse) {
      float* lp = p.lse + (((int64_t)b * p.H + cur_h) * p.M + row) * 2;
      lp[0] = (cur.m + __log2f(cur.la)) * ln2;
      lp[1] = cur.lt > 0.f ? (cur.m + __log2f(cur.lt)) * ln2 : -INFINITY;
    }
    cur_h = -1;
  };
  auto take = [&](int hh, const float* g) {
    if (cur_h != hh) {
      flush();
      cur = RowStat{g[0], g[TM], g[2 * TM]};
      cur_h = hh;
    } else {
      merge_stat(cur, g[0], g[TM], g[2 * TM]);
    }
  };
  for (int r = 0; r < cs; ++r) {
    const int i0 = r * p.per, i1 = min(i0 + p.per, p.items);
    if (i0 >= i1) break;
    const float* g = &gather[r][0][tid];
    const int h0 = i0 / p.n_kt, h1 = (i1 - 1) / p.n_kt;
    if (i0 != h0 * p.n_kt || i1 < (h0 + 1) * p.n_kt) take(h0, g + TM);
    tot += g[0];
    if (h1 != h0 && i1 != (h1 + 1) * p.n_kt) take(h1, g + 4 * TM);
  }
  flush();
  const int64_t o = (int64_t)b * p.M + row;
  const float a = p.weight * (tot / (float)p.H);
  p.A[o] = p.accumulate ? p.A[o] + a : a;
}

// How the rows and the (head, key tile) items of a call are split: clusters as
// large as they go (4 x 24 heads x 512 x 1024: 414 us in clusters of 8, 547 in
// 4); 32 rows per CTA when that still gives the SMs 1.3 CTAs each, else 16
// (measured, us with 32 / 16 rows: 256 CTAs of 32 rows 310 / 417, 512 CTAs 414 /
// 551; 104 CTAs 26.4 / 22.1, 48 CTAs 8.2 / 6.6).
struct Plan {
  int tm, cs, per;
};

Plan make_plan(int B, int H, int M, int Nk, int num_sms) {
  const int items = H * ((Nk + kTN - 1) / kTN);
  Plan pl{};
  pl.per = (items + kMaxCluster - 1) / kMaxCluster;
  pl.cs = (items + pl.per - 1) / pl.per;
  const long long ctas = (long long)B * ((M + 31) / 32) * pl.cs;
  pl.tm = 10 * ctas >= 13LL * num_sms ? 32 : 16;
  return pl;
}

template <typename T, int TM, int RM, Load kLoad>
cudaError_t launch_one(const SimtParams& p, cudaStream_t s) {
  // the shared-memory opt-in, once per device
  static int done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (!(dev >= 0 && dev < 64 && __atomic_load_n(&done[dev], __ATOMIC_ACQUIRE))) {
    e = cudaFuncSetAttribute(spatial_simt_kernel<T, TM, RM, kLoad>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)simt_smem<TM>());
    if (e == cudaSuccess) e = prefer_max_shared<spatial_simt_kernel<T, TM, RM, kLoad>>();
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) __atomic_store_n(&done[dev], 1, __ATOMIC_RELEASE);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(p.B * p.tiles * p.cs));
  cfg.blockDim = dim3(32 * (TM / RM));
  cfg.dynamicSmemBytes = simt_smem<TM>();
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)p.cs;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, spatial_simt_kernel<T, TM, RM, kLoad>, p);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <typename T, Load kLoad>
cudaError_t launch_typed(const SimtParams& p, int tm, cudaStream_t s) {
  if (tm == 32) return launch_one<T, 32, 8, kLoad>(p, s);
  return launch_one<T, 16, 4, kLoad>(p, s);
}

}  // namespace

cudaError_t launch_spatial_simt(const SpatialArgs& a, int num_sms, cudaStream_t s) {
  const Plan pl = make_plan(a.B, a.H, a.M, a.Nk, num_sms > 0 ? num_sms : 1);
  SimtParams p{};
  p.q = a.q; p.k = a.k;
  p.B = a.B; p.H = a.H; p.M = a.M; p.Nk = a.Nk; p.L = a.L; p.d = a.d;
  p.q_sb = a.q_sb; p.q_sh = a.q_sh; p.q_sn = a.q_sn;
  p.k_sb = a.k_sb; p.k_sh = a.k_sh; p.k_sn = a.k_sn;
  p.c_log2 = a.scale * 1.4426950408889634f;
  p.weight = a.weight;
  p.accumulate = a.accumulate;
  p.A = a.A; p.lse = a.lse; p.tmask = a.tmask;
  p.tiles = (a.M + pl.tm - 1) / pl.tm;
  p.n_kt = (a.Nk + kTN - 1) / kTN;
  p.items = a.H * p.n_kt;
  p.per = pl.per;
  p.cs = pl.cs;
  if ((int64_t)a.B * p.tiles * p.cs > 0x7fffffff) return cudaErrorInvalidValue;
  // 16-byte loads: d, the strides and both bases multiples of 16 bytes
  const int64_t n = a.dt == AVITS_BF16 ? 8 : 4;   // elements
  const bool vec = ((reinterpret_cast<uintptr_t>(a.q) | reinterpret_cast<uintptr_t>(a.k)) & 15u) == 0 &&
                   a.d % n == 0 && a.q_sn % n == 0 && a.k_sn % n == 0 &&
                   (a.H == 1 || (a.q_sh % n == 0 && a.k_sh % n == 0)) &&
                   (a.B == 1 || (a.q_sb % n == 0 && a.k_sb % n == 0));
  if (a.dt == AVITS_BF16)
    return vec ? launch_typed<__nv_bfloat16, kLoadVectors>(p, pl.tm, s)
               : launch_typed<__nv_bfloat16, kLoadElements>(p, pl.tm, s);
  return vec ? launch_typed<float, kLoadAsync>(p, pl.tm, s)
             : launch_typed<float, kLoadElements>(p, pl.tm, s);
}

}  // namespace avits
