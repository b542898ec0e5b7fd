// merge.cu — final merge to the dense full-resolution latent (Sec. 3.2,
// Stage 3: the remaining tokens are expanded and the sequence is laid out in
// spatial order).
//
// Nearest: full-res pixel (Y,X) of a token at (y,x) with span s takes token
// pixel ((Y-2y)/s, (X-2x)/s).  Few tokens (a batch of one): a warp, or 8 lanes, per
// token write its s x s cells in one pass; every cell is claimed by an atomicExch of
// this call's tag into a claim map in the caller's workspace (an old value equal
// to the tag = a cell covered twice).  More tokens: pass 1 writes each token's
// index into the words of its cells with plain stores, pass 2 goes over the
// cells and takes a word only if that token covers the cell in this call, so an
// entry of an earlier call is no cover.  One pass waits for a chain of round
// trips per token and for an atomic per cell; two passes are streams.
// Either way every CTA of the counting kernel adds (1 << 40) | cells to one
// 64-bit word, and the CTA whose add completes the CTA count compares the total
// with B * fh * fw (in two passes a cell covered twice makes it differ, or
// leaves a hole that pass 2 finds), then clears the word.  The map needs no
// clearing between calls.
// Bilinear (spans 1, 2 and 4): pass 1 as above with each entry carrying the
// token's level; in pass 2, where an entry that is no cover counts as a hole for
// the cells around it as well, span-1 cells are copied, coarser cells take the
// half-pixel-centred 2x bilinear resize of level 1 of the frame's pixel
// pyramid (frame_map.cuh), refined first from level 2 inside span-4 tokens.
// Algorithmic bytes: B*N*(T*elt + 12) read + B*fh*fw*T*elt written.
#include <algorithm>

#include "avits_common.cuh"
#include "avits_internal.h"
#include "frame_map.cuh"

namespace avits {
namespace {

// Workspace of the merge: a 16-byte header, then one 32-bit word per output
// cell.  Header = (tag of the last one-pass call, unused, 64-bit CTA count |
// cells), words = claim map (one pass) or cell map (two passes, bilinear).
struct MergeHeader {
  uint32_t last_tag;
  uint32_t unused;
  unsigned long long count;   // (CTAs done << 40) | cells claimed
};
constexpr int kMergeHeaderBytes = 16;

// Claim tags have bit 31 set (token indices and cell-map entries, -1 aside, have
// it clear, so a workspace used in both modes never confuses the two) and a
// 31-bit call counter in 1 .. 2^31 - 2 (never 0, the zeroed map).
__device__ __forceinline__ uint32_t next_tag(uint32_t last) {
  const uint32_t g = last & 0x7FFFFFFFu;
  return 0x80000000u | ((g == 0u || g >= 0x7FFFFFFEu) ? 1u : g + 1u);
}

// A CTA has written `cells` cells; the CTA that completes the count compares
// the total with the frame's and clears the word for the next call.
__device__ __forceinline__ void count_cells(MergeHeader* hdr, unsigned long long cells,
                                            unsigned long long frame, unsigned int* status) {
  const unsigned long long mine = (1ull << 40) | cells;
  const unsigned long long v = atomicAdd(&hdr->count, mine) + mine;
  if ((v >> 40) != (unsigned long long)gridDim.x) return;
  if ((v & ((1ull << 40) - 1ull)) != frame) raise_status(status, AVITS_ERR_COVERAGE);
  hdr->count = 0ull;
}

// Few tokens: kLanes lanes (a warp, or part of one) per token, one pass.  A token's area is known once its position and
// span are read, so the CTA's count goes out first; the claims, the count's
// atomic and the pixel loads are then in flight together and their results
// are examined last: the check adds no round trip to the copy's two
// (position, then pixels).
template <typename T, int kLanes>
__global__ void __launch_bounds__(8 * 32)
merge_nearest_warp_kernel(const T* __restrict__ mixed, int B, int N,
                          const int32_t* __restrict__ pos, const int32_t* __restrict__ span,
                          int fh, int fw, int C, T* __restrict__ out, MergeHeader* hdr,
                          uint32_t* __restrict__ claim, unsigned int* status) {
  using PV = typename Pix4<T>::V;
  constexpr int kToks = 8 * 32 / kLanes;   // per CTA
  constexpr int kStage = 8192 / kToks;     // a token of up to so many bytes takes the vector path
  pdl_wait_then_trigger();
  __shared__ __align__(16) uint8_t stage_all[kToks * kStage];
  __shared__ unsigned int cta_cells;
  if (threadIdx.x == 0) cta_cells = 0u;
  const uint32_t last = *reinterpret_cast<volatile uint32_t*>(&hdr->last_tag);
  const int lane = threadIdx.x % kLanes, slot = threadIdx.x / kLanes;
  const unsigned group = (0xffffffffu >> (32 - kLanes)) << (threadIdx.x & 31 & ~(kLanes - 1));
  const int64_t t = (int64_t)blockIdx.x * kToks + slot;
  int b = 0, y = 0, x = 0, sp = 0;
  bool valid = false;
  if (t < (int64_t)B * N) {
    b = (int)(t / N);
    y = pos[t * 2];
    x = pos[t * 2 + 1];
    sp = span[t];
    valid = !(sp <= 0 || y < 0 || x < 0 || y > fh - sp || x > fw - sp);
    if (!valid && lane == 0) raise_status(status, AVITS_ERR_COVERAGE);
  }
  __syncthreads();   // cta_cells is initialised
  if (valid && lane == 0) atomicAdd(&cta_cells, (unsigned int)(sp * sp));
  __syncthreads();
  unsigned long long v = 0ull;
  if (threadIdx.x == 0)
    v = atomicAdd(&hdr->count, (1ull << 40) | (unsigned long long)cta_cells) +
        ((1ull << 40) | (unsigned long long)cta_cells);
  const uint32_t tag = next_tag(last);
  uint32_t old0 = 0u, old1 = 0u;   // claims of cells lane and lane + kLanes
  bool twice = false;
  if (valid) {
    const int64_t base = (int64_t)b * fh * fw;
    const int area = sp * sp;
    const int T4 = C * 4;
    const T* src = mixed + t * T4;
    const int tb = T4 * (int)sizeof(T);
    const bool vec = (tb & 15) == 0 && tb <= kStage;
    uint8_t* stage = stage_all + slot * kStage;
    if (vec)
      for (int q = lane; q < tb / 16; q += kLanes)
        reinterpret_cast<uint4*>(stage)[q] = __ldg(reinterpret_cast<const uint4*>(src) + q);
    if (lane < area)
      old0 = atomicExch(&claim[base + (int64_t)(y + lane / sp) * fw + (x + lane % sp)], tag);
    if (lane + kLanes < area)
      old1 = atomicExch(
          &claim[base + (int64_t)(y + (lane + kLanes) / sp) * fw + (x + (lane + kLanes) % sp)], tag);
    for (int cell = lane + 2 * kLanes; cell < area; cell += kLanes)
      twice |= atomicExch(&claim[base + (int64_t)(y + cell / sp) * fw + (x + cell % sp)], tag) == tag;
    if (vec) {
      __syncwarp(group);
      const int cpc = tb / 16;
      for (int q = lane; q < area * cpc; q += kLanes) {
        const int cell = q / cpc, j = q - cell * cpc;
        const int u = cell / sp, w = cell - u * sp;
        const int r0 = (2 * u) / sp, r1 = (2 * u + 1) / sp;
        const int c0 = (2 * w) / sp, c1 = (2 * w + 1) / sp;
        const uint4 chunk = (sp == 1) ? reinterpret_cast<const uint4*>(stage)[j]
                                      : gather_chunk<T>(stage, j, r0, r1, c0, c1);
        const int64_t ocell = base + (int64_t)(y + u) * fw + (x + w);
        reinterpret_cast<uint4*>(out + ocell * T4)[j] = chunk;
      }
    } else {
      for (int task = lane; task < area * C; task += kLanes) {
        const int cell = task / C, c = task - cell * C;
        const int u = cell / sp, w = cell - u * sp;
        const int r0 = (2 * u) / sp, r1 = (2 * u + 1) / sp;
        const int c0 = (2 * w) / sp, c1 = (2 * w + 1) / sp;
        const T* sc = src + c * 4;
        const float p00 = load_elem(sc, r0 * 2 + c0), p01 = load_elem(sc, r0 * 2 + c1);
        const float p10 = load_elem(sc, r1 * 2 + c0), p11 = load_elem(sc, r1 * 2 + c1);
        const int64_t ocell = base + (int64_t)(y + u) * fw + (x + w);
        reinterpret_cast<PV*>(out + ocell * T4)[c] = Pix4<T>::make(p00, p01, p10, p11);
      }
    }
  }
  if (threadIdx.x == 0 && (v >> 40) == (unsigned long long)gridDim.x) {
    // every CTA has counted its cells: no cell is claimed twice unless that
    // is reported, so fewer claimed cells than cells means a hole
    if ((v & ((1ull << 40) - 1ull)) != (unsigned long long)B * fh * fw)
      raise_status(status, AVITS_ERR_COVERAGE);
    hdr->count = 0ull;
    hdr->last_tag = tag;
  }
  if (twice || old0 == tag || old1 == tag) raise_status(status, AVITS_ERR_COVERAGE);
}

// Large batches, pass 1: as merge_scatter_kernel below, for tokens of any span
// and position; the word of a cell is the token's index.  A token of more than
// 16 cells is written by its whole warp.
__global__ void __launch_bounds__(256)
merge_index_kernel(int B, int N, const int32_t* __restrict__ pos, const int32_t* __restrict__ span,
                   int fh, int fw, int32_t* __restrict__ map, MergeHeader* hdr,
                   unsigned int* status) {
  pdl_wait_then_trigger();
  __shared__ unsigned long long cta_cells;
  if (threadIdx.x == 0) cta_cells = 0ull;
  __syncthreads();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  int y = 0, x = 0, s = 0, ti = 0;
  int64_t base = 0;
  if (t < (int64_t)B * N) {
    const int b = (int)(t / N);
    ti = (int)(t - (int64_t)b * N);
    y = pos[t * 2];
    x = pos[t * 2 + 1];
    s = span[t];
    base = (int64_t)b * fh * fw;
    if (s <= 0 || y < 0 || x < 0 || y > fh - s || x > fw - s) {
      raise_status(status, AVITS_ERR_COVERAGE);
      s = 0;
    }
  }
  if (s <= 4)
    for (int u = 0; u < s; ++u)
      for (int v = 0; v < s; ++v) map[base + (int64_t)(y + u) * fw + x + v] = ti;
  for (unsigned big = __ballot_sync(0xffffffffu, s > 4); big; big &= big - 1) {
    const int src = __ffs(big) - 1;
    const int ys = __shfl_sync(0xffffffffu, y, src), xs = __shfl_sync(0xffffffffu, x, src);
    const int ss = __shfl_sync(0xffffffffu, s, src), es = __shfl_sync(0xffffffffu, ti, src);
    const int64_t bs = __shfl_sync(0xffffffffu, base, src);
    for (int u = 0; u < ss; ++u)
      for (int v = lane; v < ss; v += 32) map[bs + (int64_t)(ys + u) * fw + xs + v] = es;
  }
  unsigned long long cells = (unsigned long long)s * (unsigned long long)s;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cells += __shfl_xor_sync(0xffffffffu, cells, o);
  if (lane == 0 && cells) atomicAdd(&cta_cells, cells);
  __syncthreads();
  if (threadIdx.x == 0)
    count_cells(hdr, cta_cells, (unsigned long long)B * fh * fw, status);
}

// Large batches, pass 2: one thread per (cell, 16-byte piece of a token; one
// channel where tokens are not whole pieces), kGatherPieces of them per thread,
// reading and writing neighbouring pieces with neighbouring threads.  A cell
// whose word is not a token of this call that covers it is a hole: reported and
// not written.
constexpr int kGatherPieces = 4;

template <typename T, bool kVec>
__global__ void __launch_bounds__(256)
merge_nearest_gather_kernel(const T* __restrict__ mixed, int N, const int32_t* __restrict__ pos,
                            const int32_t* __restrict__ span, int fh, int fw, int C,
                            const int32_t* __restrict__ map, T* __restrict__ out,
                            unsigned int* status, unsigned ctas) {
  using PV = typename Pix4<T>::V;
  pdl_wait_then_trigger();
  const int T4 = C * 4;
  const unsigned parts = kVec ? (unsigned)(T4 * sizeof(T) / 16) : (unsigned)C;
  const unsigned cells = (unsigned)fh * (unsigned)fw;
  const int b = (int)(blockIdx.x / ctas);
  const unsigned g0 = (blockIdx.x - b * ctas) * (256u * kGatherPieces) + threadIdx.x;
  const int32_t* mapb = map + (int64_t)b * cells;
  const int32_t* posb = pos + (int64_t)b * N * 2;
  const int32_t* spanb = span + (int64_t)b * N;
  const T* mb = mixed + (int64_t)b * N * T4;
  unsigned cell[kGatherPieces], j[kGatherPieces];
  int t[kGatherPieces];
#pragma unroll
  for (int k = 0; k < kGatherPieces; ++k) {
    const unsigned g = g0 + k * 256u;
    cell[k] = g / parts;
    j[k] = g - cell[k] * parts;
    t[k] = cell[k] < cells ? mapb[cell[k]] : -1;
  }
  // the token's place and its piece at once: a word that is no token of this
  // call reads token 0 and is refused below
  int y[kGatherPieces], x[kGatherPieces], s[kGatherPieces];
  uint4 in[kGatherPieces];
#pragma unroll
  for (int k = 0; k < kGatherPieces; ++k) {
    if (t[k] >= N) t[k] = -1;
    const int tt = max(t[k], 0);
    y[k] = posb[(int64_t)tt * 2];
    x[k] = posb[(int64_t)tt * 2 + 1];
    s[k] = spanb[tt];
    if constexpr (kVec) in[k] = __ldg(reinterpret_cast<const uint4*>(mb + (int64_t)tt * T4) + j[k]);
  }
#pragma unroll
  for (int k = 0; k < kGatherPieces; ++k) {
    if (cell[k] >= cells) continue;
    const int Y = (int)(cell[k] / (unsigned)fw), X = (int)(cell[k] % (unsigned)fw);
    const int u = Y - y[k], w = X - x[k], sp = s[k];
    if (t[k] < 0 || u < 0 || w < 0 || u >= sp || w >= sp || y[k] < 0 || x[k] < 0 ||
        y[k] > fh - sp || x[k] > fw - sp) {
      raise_status(status, AVITS_ERR_COVERAGE);
      continue;
    }
    T* dst = out + ((int64_t)b * cells + cell[k]) * T4;
    // the token's pixel rows and columns of this cell's two
    const int r0 = (2 * u >= sp) ? 1 : 0, r1 = (2 * u + 1 >= sp) ? 1 : 0;
    const int c0 = (2 * w >= sp) ? 1 : 0, c1 = (2 * w + 1 >= sp) ? 1 : 0;
    if constexpr (kVec) {
      reinterpret_cast<uint4*>(dst)[j[k]] = sp == 1 ? in[k] : select_pixels<T>(in[k], r0, r1, c0, c1);
    } else {
      const T* sc = mb + (int64_t)t[k] * T4 + j[k] * 4;
      reinterpret_cast<PV*>(dst)[j[k]] =
          Pix4<T>::make(load_elem(sc, r0 * 2 + c0), load_elem(sc, r0 * 2 + c1),
                        load_elem(sc, r1 * 2 + c0), load_elem(sc, r1 * 2 + c1));
    }
  }
}

// The cell map starts as -1 everywhere (a hole until a token claims it).
__global__ void merge_fill_kernel(int32_t* __restrict__ map, int64_t n) {
  pdl_wait_then_trigger();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    map[i] = -1;
}

// One thread per token: its s x s cells get map_entry(token, log2 s).
__global__ void merge_map_kernel(int B, int N, const int32_t* __restrict__ pos,
                                 const int32_t* __restrict__ span, int fh, int fw,
                                 int32_t* __restrict__ map, unsigned int* status) {
  pdl_wait_then_trigger();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)B * N) return;
  const int b = (int)(t / N), ti = (int)(t % N);
  const int y = pos[t * 2], x = pos[t * 2 + 1], s = span[t];
  const int lvl = (s == 1) ? 0 : (s == 2) ? 1 : (s == 4) ? 2 : -1;
  if (lvl < 0 || y < 0 || x < 0 || y > fh - s || x > fw - s || ((y | x) & (s - 1))) {
    raise_status(status, AVITS_ERR_COVERAGE);
    return;
  }
  const int32_t entry = map_entry(ti, lvl);
  for (int u = 0; u < s; ++u)
    for (int v = 0; v < s; ++v) {
      const int old = atomicExch(&map[(int64_t)b * fh * fw + (int64_t)(y + u) * fw + x + v], entry);
      if (old != -1) raise_status(status, AVITS_ERR_COVERAGE);
    }
}

// The four pixels of a cell from the 3 x 3 level-1 pixels around it: output
// pixel row 2Y + a draws on level-1 rows (Y - 1, Y) for a = 0 and (Y, Y + 1) for
// a = 1 with weights (1/4, 3/4) / (3/4, 1/4), clamped at the frame edge by the
// neighbourhood; columns likewise.
__device__ __forceinline__ void resize_cell(const float (&lv)[3][3], float (&r)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int a = q >> 1, b = q & 1;
    r[q] = bil_combine(lv[a][b], lv[a][b + 1], lv[a + 1][b], lv[a + 1][b + 1], a ? 0.75f : 0.25f,
                       a ? 0.25f : 0.75f, b ? 0.75f : 0.25f, b ? 0.25f : 0.75f);
  }
}

// Bilinear merge, pass 1.  One thread per token: its s x s cells get
// map_entry(token, log2 s) by plain stores into a map that still holds the
// entries of earlier calls; the CTAs add up the cells written as the nearest
// merge does.  Pass 2 takes an entry only if its token covers the cell, so a
// cell nothing wrote in this call is found there; a double cover makes the
// total differ, or leaves such a cell.  That needs neither a fill of the map
// nor atomics on its cells.
__global__ void __launch_bounds__(256)
merge_scatter_kernel(int B, int N, const int32_t* __restrict__ pos,
                     const int32_t* __restrict__ span, int fh, int fw,
                     int32_t* __restrict__ map, MergeHeader* hdr, unsigned int* status) {
  pdl_wait_then_trigger();
  __shared__ unsigned int cta_cells;
  if (threadIdx.x == 0) cta_cells = 0u;
  __syncthreads();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned int cells = 0u;
  if (t < (int64_t)B * N) {
    const int b = (int)(t / N), ti = (int)(t - (int64_t)b * N);
    const int y = pos[t * 2], x = pos[t * 2 + 1], s = span[t];
    const int lvl = (s == 1) ? 0 : (s == 2) ? 1 : (s == 4) ? 2 : -1;
    if (lvl < 0 || y < 0 || x < 0 || y > fh - s || x > fw - s || ((y | x) & (s - 1))) {
      raise_status(status, AVITS_ERR_COVERAGE);
    } else {
      const int32_t entry = map_entry(ti, lvl);
      int32_t* m = map + (int64_t)b * fh * fw + (int64_t)y * fw + x;
      for (int u = 0; u < s; ++u)
        for (int v = 0; v < s; ++v) m[(int64_t)u * fw + v] = entry;
      cells = (unsigned int)(s * s);
    }
  }
  cells = __reduce_add_sync(0xffffffffu, cells);
  if ((threadIdx.x & 31) == 0 && cells) atomicAdd(&cta_cells, cells);
  __syncthreads();
  if (threadIdx.x == 0) count_cells(hdr, cta_cells, (unsigned long long)B * fh * fw, status);
}

// What pass 1 left for a cell: its word and the place of the token that the
// word names (token 0 where it names none of this call's; loaded at once, so that
// a caller can have several in flight).
struct CellWord {
  int32_t e;
  int s, y, x;
  __device__ void place(int N, const int32_t* __restrict__ posb, const int32_t* __restrict__ spanb) {
    const int t = e >= 0 && map_tok(e) < N ? map_tok(e) : 0;
    s = spanb[t];
    y = posb[t * 2];
    x = posb[t * 2 + 1];
  }
  // The word if its token covers the cell in this call, else -1 (a hole: the
  // word is what an earlier call, of either mode and of any token count, left
  // there).  Only a word that passed here may be followed to a token.
  __device__ int32_t live(int N, int fh, int fw, int Y, int X) const {
    const bool ok = e >= 0 && map_lvl(e) <= kMaxMapLevel && map_tok(e) < N && s == 1 << map_lvl(e) &&
                    (Y & ~(s - 1)) == y && (X & ~(s - 1)) == x && y <= fh - s && x <= fw - s;
    return ok ? e : -1;
  }
};

// Pass 1b for merge_bilinear_kernel, whose channels read a cell's word many
// times over: words that no token of this call stands behind become -1.
__global__ void __launch_bounds__(256)
merge_live_kernel(int64_t ncell, int N, const int32_t* __restrict__ pos,
                  const int32_t* __restrict__ span, int fh, int fw, int32_t* __restrict__ map) {
  pdl_wait_then_trigger();
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= ncell) return;
  CellWord w{map[g]};
  if (w.e < 0) return;
  const int cells = fh * fw;
  const int b = (int)(g / cells), cell = (int)(g % cells);
  w.place(N, pos + (int64_t)b * N * 2, span + (int64_t)b * N);
  if (w.live(N, fh, fw, cell / fw, cell % fw) < 0) map[g] = -1;
}

// Bilinear merge, pass 2, one thread per (output cell, channel): tokens whose
// rows are not whole 16-byte pieces.  Every word of the map is live or negative
// (merge_live_kernel).  A hole is reported and gives zeros, a span-1 cell is
// copied, a coarser cell's four pixels are the 2x bilinear resize of the level-1
// pixels around it (a 3 x 3 neighbourhood, clamped to the frame): the frame's
// own, or inside a span-4 token the 2x resize of level 2 (the coarse-to-fine
// cascade; spans are at most 4).
template <typename T>
__global__ void
merge_bilinear_kernel(const T* __restrict__ mixed, int B, int N, int fh, int fw, int C,
                      const int32_t* __restrict__ map, T* __restrict__ out, unsigned int* status) {
  using PV = typename Pix4<T>::V;
  pdl_wait_then_trigger();
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t cells = (int64_t)fh * fw;
  if (g >= (int64_t)B * cells * C) return;
  const int c = (int)(g % C);
  const int64_t bc = g / C;
  const int b = (int)(bc / cells);
  const int cell = (int)(bc % cells);
  const int Y = cell / fw, X = cell - Y * fw;
  const int T4 = C * 4;
  const int32_t* mapb = map + (int64_t)b * cells;
  const T* mb = mixed + (int64_t)b * N * T4;
  const int32_t e = mapb[cell];
  PV* dst = reinterpret_cast<PV*>(out + bc * T4) + c;
  if (e < 0) {
    raise_status(status, AVITS_ERR_COVERAGE);
    *dst = Pix4<T>::make(0.f, 0.f, 0.f, 0.f);
    return;
  }
  if (map_lvl(e) == 0) {
    *dst = reinterpret_cast<const PV*>(mb + (int64_t)map_tok(e) * T4)[c];
    return;
  }
  int rr[3], cc[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    rr[k] = min(max(Y - 1 + k, 0), fh - 1);
    cc[k] = min(max(X - 1 + k, 0), fw - 1);
  }
  float lv[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int32_t en = mapb[(int64_t)rr[i] * fw + cc[j]];
      lv[i][j] = (en >= 0 && map_lvl(en) >= 2)
                     ? frame_resize2x(2, mb, T4, mapb, fh, fw, c, rr[i], cc[j])
                     : frame_pixel<1>(mb, T4, mapb, fw, c, rr[i], cc[j]);
    }
  float r[4];
  resize_cell(lv, r);
  *dst = Pix4<T>::make(r[0], r[1], r[2], r[3]);
}

// Bilinear merge, pass 2, for tokens of whole 16-byte pieces: a CTA takes a tile
// of 16 x 16 cells and two pieces (32 bytes) of the channels.  It loads the
// cell map of the tile and four cells around it (a word that no token of this
// call stands behind is a hole: zeros, and reported within the tile), turns every
// cell of the tile and the ring next to it into its level-1 pixel (one 16-byte
// load: a span-2
// token's pixel, or the average of a span-1 token's four) in shared memory,
// and writes the cells from the 3 x 3 level-1 pixels around them; span-1 cells
// are copied.  Only where a span-4 token is near does it also build the level-2
// pixels (from the wider ring) and refine the level-1 pixels inside such
// tokens.  Every value is the one merge_bilinear_kernel would compute, in the same
// order of operations.  What bounds it: the chain map - token - shared memory -
// cell at a few CTAs per SM, then the copies.  us of the two kernels, against a
// thread per (cell, channel) behind a fill and an atomic scatter, bf16, 64 x 64
// cells of 16 channels: batch 1 8.5 -> 6.0, 16 31.7 -> 11.9, 64 103 -> 32.2; batch 64
// with spans 1, 2 and 4 5371 -> 49.3 (a value of level 2 was pooled anew by every
// thread that drew on it).  Words are checked where the map is loaded, the wider
// ring's as well, a thread's three words and then their tokens' places in flight
// together (one after the other: 6.7, 13.0, 33.8 and 60.7).  Left out: a thread
// per 2 x 2 cells with the neighbourhood in registers, 10.5 at batch 16 but 5580
// with span 4; three pieces of a thread in flight (13.2 against 12.8); four pieces
// per CTA (12.9); the pieces' planes 16 banks apart (12.4).
constexpr int kTile = 16;
constexpr int kHalo = 4;                        // cells around the tile that level 2 can draw on
constexpr int kReg = kTile + 2 * kHalo;
constexpr int kTilePieces = 2;

template <typename T>
__global__ void __launch_bounds__(256)
merge_bilinear_tile_kernel(const T* __restrict__ mixed, int N, const int32_t* __restrict__ pos,
                           const int32_t* __restrict__ span, int fh, int fw, int C,
                           const int32_t* __restrict__ map, T* __restrict__ out,
                           unsigned int* status, unsigned tiles_x, unsigned tiles_y,
                           unsigned groups) {
  constexpr int kCh = Chunk<T>::kCh;
  __shared__ int32_t smap[kReg][kReg];
  __shared__ float l1[kTilePieces][kCh][kReg][kReg];
  __shared__ float l2[kTilePieces][kCh][kReg / 2][kReg / 2];
  pdl_wait_then_trigger();
  unsigned blk = blockIdx.x;
  const int grp = (int)(blk % groups);
  blk /= groups;
  const int X0 = (int)(blk % tiles_x) * kTile;
  blk /= tiles_x;
  const int Y0 = (int)(blk % tiles_y) * kTile, b = (int)(blk / tiles_y);
  const int T4 = C * 4, cpc = C / kCh;
  const int npc = min(kTilePieces, cpc - grp * kTilePieces);   // pieces of this CTA
  const int32_t* mapb = map + (int64_t)b * fh * fw;
  const int32_t* posb = pos + (int64_t)b * N * 2;
  const int32_t* spanb = span + (int64_t)b * N;
  const T* mb = mixed + (int64_t)b * N * T4;
  T* ob = out + (int64_t)b * fh * fw * T4;
  // the map, -1 off the frame and for words that no token of this call stands
  // behind; all of a thread's words, then all of their tokens' places in flight
  constexpr int kWords = (kReg * kReg + 255) / 256;
  CellWord cw[kWords];
#pragma unroll
  for (int k = 0; k < kWords; ++k) {
    const int i = threadIdx.x + 256 * k, Y = Y0 - kHalo + i / kReg, X = X0 - kHalo + i % kReg;
    cw[k].e = i < kReg * kReg && Y >= 0 && Y < fh && X >= 0 && X < fw ? mapb[(int64_t)Y * fw + X] : -1;
  }
#pragma unroll
  for (int k = 0; k < kWords; ++k) cw[k].place(N, posb, spanb);
  bool wide = false;   // a span-4 token in the tile or the ring next to it
#pragma unroll
  for (int k = 0; k < kWords; ++k) {
    const int i = threadIdx.x + 256 * k, r = i / kReg, c = i % kReg;
    if (i >= kReg * kReg) break;
    const int Y = Y0 - kHalo + r, X = X0 - kHalo + c;
    const int32_t e = cw[k].live(N, fh, fw, Y, X);
    if (e < 0 && r >= kHalo && r < kHalo + kTile && c >= kHalo && c < kHalo + kTile && Y < fh && X < fw)
      raise_status(status, AVITS_ERR_COVERAGE);
    smap[r][c] = e;
    wide = wide || (e >= 0 && map_lvl(e) >= 2 && r >= kHalo - 1 && r <= kHalo + kTile &&
                    c >= kHalo - 1 && c <= kHalo + kTile);
  }
  wide = __syncthreads_or(wide);
  auto piece = [&](int32_t e, int pc) {
    return *(reinterpret_cast<const uint4*>(mb + (int64_t)map_tok(e) * T4) + grp * kTilePieces + pc);
  };
  auto write = [&](int Y, int X, int pc, const uint4& w) {
    *(reinterpret_cast<uint4*>(ob + ((int64_t)Y * fw + X) * T4) + grp * kTilePieces + pc) = w;
  };
  // level-1 pixels of the cells outside span-4 tokens; span-1 cells and holes of
  // the tile are written here
  const int first = wide ? 0 : kHalo - 1, side = wide ? kReg : kTile + 2;
  for (int i = threadIdx.x; i < side * side * kTilePieces; i += 256) {
    const int pc = i % kTilePieces, q = i / kTilePieces;
    const int r = first + q / side, c = first + q % side;
    if (pc >= npc) continue;
    const int32_t e = smap[r][c];
    const int Y = Y0 - kHalo + r, X = X0 - kHalo + c;
    const bool mine = r >= kHalo && r < kHalo + kTile && c >= kHalo && c < kHalo + kTile &&
                      Y < fh && X < fw;
    const uint4 w = e >= 0 ? piece(e, pc) : make_uint4(0u, 0u, 0u, 0u);
    const int lvl = e >= 0 ? map_lvl(e) : -1;
    if (mine && lvl <= 0) write(Y, X, pc, w);   // a span-1 cell, or zeros in a hole
    float p[kCh][4];
    Chunk<T>::unpack(w, p);
#pragma unroll
    for (int ch = 0; ch < kCh; ++ch) {
      float v = 0.f;
      if (lvl == 0)
        v = __fmul_rn(__fadd_rn(__fadd_rn(p[ch][0], p[ch][1]), __fadd_rn(p[ch][2], p[ch][3])),
                      0.25f);
      else if (lvl == 1)
        v = (Y & 1) ? ((X & 1) ? p[ch][3] : p[ch][2]) : ((X & 1) ? p[ch][1] : p[ch][0]);
      l1[pc][ch][r][c] = v;
    }
  }
  __syncthreads();
  if (wide) {
    // level 2: a span-4 token's pixel, or the average of four level-1 pixels
    for (int i = threadIdx.x; i < (kReg / 2) * (kReg / 2) * kTilePieces; i += 256) {
      const int pc = i % kTilePieces, q = i / kTilePieces;
      const int r = q / (kReg / 2), c = q % (kReg / 2);
      if (pc >= npc) continue;
      const int32_t e = smap[2 * r][2 * c];
      const bool four = e >= 0 && map_lvl(e) >= 2;
      float p[kCh][4];
      if (four) Chunk<T>::unpack(piece(e, pc), p);
      const int R = (Y0 - kHalo) / 2 + r, Q = (X0 - kHalo) / 2 + c;
#pragma unroll
      for (int ch = 0; ch < kCh; ++ch) {
        const float(*s)[kReg] = l1[pc][ch];
        l2[pc][ch][r][c] =
            four ? ((R & 1) ? ((Q & 1) ? p[ch][3] : p[ch][2]) : ((Q & 1) ? p[ch][1] : p[ch][0]))
            : e < 0 ? 0.f
                    : __fmul_rn(__fadd_rn(__fadd_rn(s[2 * r][2 * c], s[2 * r][2 * c + 1]),
                                          __fadd_rn(s[2 * r + 1][2 * c], s[2 * r + 1][2 * c + 1])),
                                0.25f);
      }
    }
    __syncthreads();
    // level 1 inside span-4 tokens: the 2x resize of level 2
    for (int i = threadIdx.x; i < (kTile + 2) * (kTile + 2) * kTilePieces; i += 256) {
      const int pc = i % kTilePieces, q = i / kTilePieces;
      const int r = kHalo - 1 + q / (kTile + 2), c = kHalo - 1 + q % (kTile + 2);
      const int32_t e = smap[r][c];
      if (pc >= npc || e < 0 || map_lvl(e) < 2) continue;
      int r0, r1, c0, c1;
      float wy0, wy1, wx0, wx1;
      bil_axis(Y0 - kHalo + r, fh / 2, r0, r1, wy0, wy1);
      bil_axis(X0 - kHalo + c, fw / 2, c0, c1, wx0, wx1);
      r0 -= (Y0 - kHalo) / 2;
      r1 -= (Y0 - kHalo) / 2;
      c0 -= (X0 - kHalo) / 2;
      c1 -= (X0 - kHalo) / 2;
#pragma unroll
      for (int ch = 0; ch < kCh; ++ch)
        l1[pc][ch][r][c] = bil_combine(l2[pc][ch][r0][c0], l2[pc][ch][r0][c1], l2[pc][ch][r1][c0],
                                       l2[pc][ch][r1][c1], wy0, wy1, wx0, wx1);
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < kTile * kTile * kTilePieces; i += 256) {
    const int pc = i % kTilePieces, q = i / kTilePieces;
    const int r = kHalo + q / kTile, c = kHalo + q % kTile;
    const int32_t e = smap[r][c];
    const int Y = Y0 - kHalo + r, X = X0 - kHalo + c;
    if (pc >= npc || e < 0 || map_lvl(e) == 0 || Y >= fh || X >= fw) continue;
    float v[kCh][4];
#pragma unroll
    for (int ch = 0; ch < kCh; ++ch) {
      float lv[3][3];
#pragma unroll
      for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int w = 0; w < 3; ++w)
          lv[u][w] = l1[pc][ch][r + (min(max(Y - 1 + u, 0), fh - 1) - Y)]
                               [c + (min(max(X - 1 + w, 0), fw - 1) - X)];
      resize_cell(lv, v[ch]);
    }
    write(Y, X, pc, Chunk<T>::pack(v));
  }
}

// One pass, a warp per token, up to here: us in one / two passes at 1945 tokens
// 3.2 / 4.0, 3040 4.0 / 4.5, 3890 5.4 / 4.5, 7780 7.1 / 4.4, 124480 99 / 12.4 (64 x 64
// cells per 1945 tokens, bf16, 16 channels: 270 bytes of output per token).  The
// second line holds for tokens of up to so many bytes of output (12 fp32 channels,
// 404 bytes, 3040 tokens: 5.1 / 4.4).
constexpr int kOnePassTokensPerSm = 16;
constexpr int kOnePassMoreTokensPerSm = 20;
constexpr int kOnePassMoreBytes = 288;
// Then 8 lanes per token while its output is small, where two passes are two
// chains of latency: us with 8 lanes / two passes, 64 x 64 cells per 1945 tokens, 4
// bf16 channels (67 bytes of output per token) 3890 tokens 3.2 / 4.6, 9725 3.7 / 4.8;
// 8 channels (135) 3.6 / 4.6, 4.0 / 4.7; 16 channels (270) 4.0 / 4.5, 4.85 / 4.8.  With
// spans up to 4 a few tokens have most of the cells: 4 channels (108) 3648 tokens 4.0
// / 4.7, 9728 4.9 / 4.8; 8 channels (216) 5.3 / 4.8, 6.3 / 4.95.
constexpr int kOnePassLanes = 8;
constexpr int kOnePassSmallTokensPerSm = 64;
constexpr int kOnePassSmallBytes = 144;
constexpr int64_t kMaxWork = 0xfffffff0ll - 1024;   // 32-bit indices within an element
constexpr int64_t kMaxGrid = 0x7fffffffll;

template <typename T>
cudaError_t launch_t(const void* mixed, int B, int N, const int32_t* pos, const int32_t* span,
                     int fh, int fw, int C, avits_upmode mode, void* out, void* ws,
                     unsigned int* status, cudaStream_t s) {
  MergeHeader* hdr = static_cast<MergeHeader*>(ws);
  uint32_t* words = reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(ws) + kMergeHeaderBytes);
  if (mode == AVITS_UP_NEAREST) {
    const int64_t ntok = (int64_t)B * N;
    int dev = 0, sms = 0;
    cudaError_t e0 = cudaGetDevice(&dev);
    if (e0 == cudaSuccess) e0 = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e0 != cudaSuccess) return e0;
    cudaError_t e = prefer_max_shared<merge_nearest_warp_kernel<T, 32>>();
    if (e == cudaSuccess) e = prefer_max_shared<merge_nearest_warp_kernel<T, kOnePassLanes>>();
    if (e == cudaSuccess) e = prefer_max_shared<merge_index_kernel>();
    if (e == cudaSuccess) e = prefer_max_shared<merge_nearest_gather_kernel<T, true>>();
    if (e == cudaSuccess) e = prefer_max_shared<merge_nearest_gather_kernel<T, false>>();
    if (e != cudaSuccess) return e;
    const bool whole = (C * 4 * (int)sizeof(T)) % 16 == 0;
    const int64_t work = (int64_t)fh * fw * (whole ? C * 4 * (int)sizeof(T) / 16 : C);
    // one pass (latency-bound sizes)
    const auto up_to = [&](int per_sm) { return ntok <= (int64_t)std::max(1, sms) * per_sm; };
    const int64_t out_bytes = (int64_t)B * fh * fw * C * 4 * (int)sizeof(T);
    const bool few = up_to(kOnePassTokensPerSm) ||
                     (up_to(kOnePassMoreTokensPerSm) && out_bytes <= ntok * kOnePassMoreBytes) ||
                     work > kMaxWork || B * ((work + 255) / 256) > kMaxGrid;
    const bool small = up_to(kOnePassSmallTokensPerSm) && out_bytes <= ntok * kOnePassSmallBytes;
    if (few || small) {
      const int toks = few ? 8 : 8 * 32 / kOnePassLanes;
      e = launch_pdl(few ? merge_nearest_warp_kernel<T, 32>
                         : merge_nearest_warp_kernel<T, kOnePassLanes>,
                     dim3((unsigned)((ntok + toks - 1) / toks)), dim3(8 * 32), 0, s,
                     static_cast<const T*>(mixed), B, N, pos, span, fh, fw, C,
                     static_cast<T*>(out), hdr, words, status);
      if (e != cudaSuccess) return e;
      return cudaGetLastError();
    }
    int32_t* map = reinterpret_cast<int32_t*>(words);
    e = launch_pdl(merge_index_kernel, dim3((unsigned)((ntok + 255) / 256)), dim3(256), 0, s, B, N,
                   pos, span, fh, fw, map, hdr, status);
    if (e != cudaSuccess) return e;
    const unsigned ctas = (unsigned)((work + 256 * kGatherPieces - 1) / (256 * kGatherPieces));
    e = launch_pdl(whole ? merge_nearest_gather_kernel<T, true> : merge_nearest_gather_kernel<T, false>,
                   dim3(ctas * (unsigned)B), dim3(256), 0, s, static_cast<const T*>(mixed), N, pos,
                   span, fh, fw, C, static_cast<const int32_t*>(map), static_cast<T*>(out), status,
                   ctas);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
  }
  // two kernels (scatter of the cell map, gather; where tokens are not whole
  // 16-byte pieces a third between them), each a programmatic dependent of the
  // one before
  int32_t* map = reinterpret_cast<int32_t*>(words);
  const int64_t nt = (int64_t)B * N;
  cudaError_t e = prefer_max_shared<merge_scatter_kernel>();
  if (e == cudaSuccess) e = prefer_max_shared<merge_live_kernel>();
  if (e == cudaSuccess) e = prefer_max_shared<merge_bilinear_kernel<T>>();
  if (e == cudaSuccess) e = prefer_max_shared<merge_bilinear_tile_kernel<T>>();
  if (e != cudaSuccess) return e;
  e = launch_pdl(merge_scatter_kernel, dim3((unsigned)((nt + 255) / 256)), dim3(256), 0, s, B, N,
                 pos, span, fh, fw, map, hdr, status);
  if (e != cudaSuccess) return e;
  const bool whole = (C * 4 * (int)sizeof(T)) % 16 == 0;
  const int64_t ty = (fh + kTile - 1) / kTile, tx = (fw + kTile - 1) / kTile;
  const int64_t groups = (C / Chunk<T>::kCh + kTilePieces - 1) / kTilePieces;
  if (whole && B * ty * tx * groups <= kMaxGrid) {
    e = launch_pdl(merge_bilinear_tile_kernel<T>, dim3((unsigned)(B * ty * tx * groups)), dim3(256),
                   0, s, static_cast<const T*>(mixed), N, pos, span, fh, fw, C,
                   static_cast<const int32_t*>(map), static_cast<T*>(out), status, (unsigned)tx,
                   (unsigned)ty, (unsigned)groups);
  } else {
    const int64_t ncell = (int64_t)B * fh * fw, all = ncell * C;
    e = launch_pdl(merge_live_kernel, dim3((unsigned)((ncell + 255) / 256)), dim3(256), 0, s, ncell,
                   N, pos, span, fh, fw, map);
    if (e != cudaSuccess) return e;
    e = launch_pdl(merge_bilinear_kernel<T>, dim3((unsigned)((all + 255) / 256)), dim3(256), 0, s,
                   static_cast<const T*>(mixed), B, N, fh, fw, C, static_cast<const int32_t*>(map),
                   static_cast<T*>(out), status);
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_cell_map(int B, int N, const int32_t* pos, const int32_t* span, int fh, int fw,
                            int32_t* map, unsigned int* status, cudaStream_t s) {
  const int64_t ncell = (int64_t)B * fh * fw;
  cudaError_t e = prefer_max_shared<merge_fill_kernel>();
  if (e == cudaSuccess) e = prefer_max_shared<merge_map_kernel>();
  if (e != cudaSuccess) return e;
  const int fill_grid = (int)std::min<int64_t>((ncell + 255) / 256, 1024);
  e = launch_pdl(merge_fill_kernel, dim3(fill_grid), dim3(256), 0, s, map, ncell);
  if (e != cudaSuccess) return e;
  const int64_t nt = (int64_t)B * N;
  e = launch_pdl(merge_map_kernel, dim3((unsigned)((nt + 255) / 256)), dim3(256), 0, s, B, N, pos,
                 span, fh, fw, map, status);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

size_t merge_workspace_bytes(int B, int fh, int fw) {
  return kMergeHeaderBytes + sizeof(uint32_t) * (size_t)B * fh * fw;
}

cudaError_t launch_merge(const void* mixed, avits_dtype dt, int B, int N, const int32_t* pos,
                         const int32_t* span, int fh, int fw, int C, avits_upmode mode,
                         void* out, void* ws, unsigned int* status, cudaStream_t s) {
  if (dt == AVITS_BF16)
    return launch_t<__nv_bfloat16>(mixed, B, N, pos, span, fh, fw, C, mode, out, ws, status, s);
  return launch_t<float>(mixed, B, N, pos, span, fh, fw, C, mode, out, ws, status, s);
}

}  // namespace avits
