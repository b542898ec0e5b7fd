// attention_tc.cu — the joint-attention forward of a double-stream block
// (Eq. 4-5, Sec. 3.3.1) on the sm_103a tensor cores, with the spatial score
// of Eq. 3 read off the same softmax.
//
// For batch b, head h and query row i of the joint sequence [C; Z]:
//   O_i      = sum_j softmax_j(scale * q_i . k_j) v_j        (all Nk keys)
//   lse_i    = log sum_j exp(scale * q_i . k_j), over all keys and over the
//              text keys (the first L)
//   A_i     (+)= weight * mean_h exp(lse_txt_i - lse_all_i)  (Eq. 5, Eq. 3)
// The text mass Eq. 5 extracts is a by-product of the softmax the block
// computes anyway: the only extra work is one running sum per row.
//
// Work decomposition (persistent, one CTA per SM): unit = (b, h, 256 query
// rows = two 128-row tiles); CTA c takes units c, c + grid, ...  Each unit
// runs over all key tiles (128 keys), so O and the row statistics stay in
// the CTA and no partial results cross CTAs (except Eq. 3's head sum).
//
// Tensor memory (512 columns): S_t (128 columns per query tile), whose first
// 64 columns are overwritten by P_t (bf16 pairs) as the softmax goes, and O_t
// (D columns per tile).  S_t(g+1) is issued right behind the PV product that
// reads P_t(g), by the same thread, so the two never overlap; while one tile's
// softmax runs, the tensor pipe works on the other tile's PV and S.
//
// Roles (12 warps):
//   warp 0       TMA producer: Q tiles, then the K and V tiles through a
//                4-stage ring (8 at d = 64) in the order the MMAs consume them
//                (K_0, V_0, K_1, V_1, ...), 128-byte swizzle.
//   warps 1, 2   MMA issuers of query tile 0 / 1 (warp 1 owns tensor
//                memory), in turns: O_t += P_t(g) V_g (A = P_t from tensor
//                memory, the tcgen05.mma TS form; V read in its natural
//                [keys, d] layout as an MN-major shared-memory operand, no
//                transpose copy) in two 64-key halves, each as soon as its
//                half of P is written, then S_t(g+1) = Q_t K_(g+1)^T.  The
//                turns keep the tiles half a period apart: without them both
//                softmaxes ran at the same time, shared the MUFU, and then
//                both waited for the pipe (4570 clocks per key tile).  A warp
//                waits for its operands during the other's turn: a wait costs
//                it ~190 clocks even when the barrier has completed, and one
//                warp issuing for both tiles spent 3600 clocks per key tile
//                on six of them.
//   warp 3       no role.
//   warps 4-7    softmax and epilogue of query tile 0, warps 8-11 of tile 1:
//                one row per thread (TMEM lane), 64 keys at a time:
//                exponentials against the running reference m (packed FMA +
//                MUFU), the fp32 sums over all keys and over the text keys
//                (the only addition the score needs), the bf16 P half to
//                tensor memory.  The row maximum is not taken on this path
//                (it cost 480 of a tile's 2300 clocks): m is the maximum of
//                the row's first key tile and moves, to a half's maximum, only
//                when that half's sum reaches 2^16 (or is NaN); l and O are
//                then rescaled.  The epilogue divides O by the row sum and
//                stores it 64 columns at a time through a swizzled staging
//                block with a bulk tensor copy.  These warps take 208
//                registers, the others 88 (at 168 each the compiler spilled).
//
// What bounds it: the chain of one tile's step, S product and its completion
// (~900 clocks; 8 products whose operands leave shared memory at its 128 bytes
// a clock), two halves of load, exponentials and store (~1600), waits (~200),
// the second half's PV product; the pipe itself needs ~2290 clocks per key tile
// for both tiles.  24 heads of 128, one image at 1024^2 (1536 x 1536): 27.2 ->
// 26.2 us; at 2048^2 (4608 x 4608): 197 -> 178 us (1462 TFLOP/s, 0.76 of the
// measured bf16 peak); batch 2: 395 -> 354 us, 413 -> 375 where logits rise along
// the keys.  Without the care for P's rounding (kBig) 23.8 / 164 / 327 us, but the
// error of O against 64 bits was then 3 to 6 % above the earlier kernel's; with
// it 1 to 4 % below (from 2^7 on: 0.5 to 2 % below, 25.7 / 175 / 349 us; 2^5: 1 to
// 6 %, 362 us; always: 7 to 11 %, 385 us).  References moved from 2^9 on instead:
// equal, 370 us.
// Measured and left out at 2048^2 (against 164): 16 softmax warps, two threads
// per row (186 us); S in 64-key products with the next step's S behind this
// step's PV (186: half-width products read Q twice); the turn passed before the
// S product is issued (192); a jumped row's redo as a loop around the half (228).
// Every wait is bounded (avits_common.cuh); after a timeout every role skips
// its remaining work, drains what it issued and the CTA releases tensor
// memory and exits.
#include <cuda.h>

#include "avits_common.cuh"
#include "avits_internal.h"
#include "tc_common.cuh"

namespace avits {
namespace {

using namespace tc;

constexpr int kBM = 128;            // query rows per tile (= TMEM lanes)
constexpr int kBN = 128;            // keys per tile
constexpr int kQTiles = 2;          // query tiles per unit
constexpr int kUnitRows = kBM * kQTiles;
constexpr int kThreads = 12 * 32;
constexpr int kTmemCols = 512;
constexpr int kHalf = kBN / 2;      // keys the softmax handles at a time
constexpr float kJump = 0x1p16f;    // a half's sum from which the reference moves
constexpr float kBig = 0x1p6f;      // and from which P's rounding is made up for
constexpr uint32_t kIdescS = idesc_bf16(kBM, kBN, false);

template <int D>
struct Cfg {
  static constexpr int kCB = D / 64;                   // 128-byte column blocks per row
  static constexpr int kTileBytes = kCB * kBM * 128;   // one 128-row bf16 tile
  static constexpr int kStages = (D == 128) ? 4 : 8;   // K / V ring
  static constexpr int kQBytes = kQTiles * kTileBytes;
  static constexpr int kKVBytes = kStages * kTileBytes;
  static constexpr uint32_t kIdescPV = idesc_bf16(kBM, D, true);
};
// O staging at a unit's end: per query tile one 128-row x 64-column bf16
// block (128-byte swizzle), stored with a bulk tensor copy per 64 columns
constexpr int kStageTileBytes = kBM * 128;
constexpr int kStageBytes = kQTiles * kStageTileBytes;
constexpr int kMaxStages = 8;
// Tensor memory columns: S_t (P_t in the first half of its columns), then O_t.
constexpr int kColS = 0, kColO = kQTiles * kBN;

struct Bars {
  uint64_t q_full[kQTiles], q_empty[kQTiles];
  uint64_t kv_full[kMaxStages], kv_empty[kMaxStages];
  uint64_t s_full[kQTiles], p_full[kQTiles][2], pv_half[kQTiles];
  uint64_t o_full[kQTiles], o_empty[kQTiles], turn[kQTiles], drain[kQTiles];
  uint32_t tmem_base;
  int abort;
};

template <int D>
constexpr int smem_bytes() {
  return Cfg<D>::kQBytes + Cfg<D>::kKVBytes + kStageBytes + (int)sizeof(Bars) + 1024;
}

struct AttnParams {
  int B, H, Mq, Nk, L;
  int n_qp, n_kt, n_units;
  float c_log2, weight;
  int accumulate;
  float* A;                   // [B,Mq] or NULL
  float* lse;                 // [B,H,Mq,2] or NULL
  unsigned long long* acc;    // [B][n_qp * 256] head-sum words (A != NULL)
  int rows_pad;
  unsigned int* status;
};

// WG-wide AND of v over the `count` threads of named barrier `id`.
__device__ __forceinline__ bool bar_and(int id, int count, bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(id), "r"(count)
      : "memory");
  return r != 0;
}

// Row maximum of 64 S columns whose first key is key0; with kGeneral keys >= Nk
// are left out.
template <bool kGeneral>
__device__ __forceinline__ float half_max(const uint32_t (&a)[32], const uint32_t (&b)[32],
                                          int key0, int Nk) {
  float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
  for (int e = 0; e < 32; ++e) {
    float x = __uint_as_float(a[e]), y = __uint_as_float(b[e]);
    if (kGeneral && key0 + e >= Nk) x = -INFINITY;
    if (kGeneral && key0 + 32 + e >= Nk) y = -INFINITY;
    m[e & 3] = max3(m[e & 3], x, y);
  }
  return fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
}

// O_t row *= f (D fp32 columns at tO), 64 columns at a time.
template <int D>
__device__ __forceinline__ void rescale_o(uint32_t tO, float f) {
#pragma unroll 1
  for (int k = 0; k < D; k += 64) {
    uint32_t a[32], b[32];
    tmem_ld64_wait(tO + (uint32_t)k, a, b);
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      a[e] = __float_as_uint(__uint_as_float(a[e]) * f);
      b[e] = __float_as_uint(__uint_as_float(b[e]) * f);
    }
    tmem_st32(tO + (uint32_t)k, a);
    tmem_st32(tO + (uint32_t)k + 32, b);
  }
}

// Exponentials of 64 S columns (a: the first 32, b: the next; first key key0)
// against the reference m, their fp32 sum, the sum over the text keys, and the
// bf16 numerators: w[i] = keys 2i, 2i + 1 (the even key in the low half), the
// layout the PV product reads P_t in from tensor memory.  kGeneral: keys
// beyond Nk give 0 and text keys are counted one by one (else all 64 keys are
// valid, and text keys or not).
template <bool kGeneral>
__device__ __forceinline__ void exp_half(const uint32_t (&a)[32], const uint32_t (&b)[32],
                                         uint32_t (&w)[32], int key0, int Nk, int L, float c,
                                         float m, float& sum, float& text) {
  const float nm = -m;
  float s[4] = {0.f, 0.f, 0.f, 0.f}, t = 0.f;
#pragma unroll
  for (int e = 0; e < 64; e += 2) {
    const uint32_t r0 = e < 32 ? a[e & 31] : b[e & 31], r1 = e < 32 ? a[(e & 31) + 1] : b[(e & 31) + 1];
    float x0, x1;
    ffma2(__uint_as_float(r0), __uint_as_float(r1), c, nm, x0, x1);
    float e0 = ex2(x0), e1 = ex2(x1);
    if (kGeneral) {
      if (key0 + e >= Nk) e0 = 0.f;
      if (key0 + e + 1 >= Nk) e1 = 0.f;
      if (key0 + e < L) t += e0;
      if (key0 + e + 1 < L) t += e1;
    }
    fadd2(s[(e & 2)], s[(e & 2) + 1], e0, e1);
    w[e >> 1] = pack_bf16x2(e0, e1);
  }
  sum = (s[0] + s[1]) + (s[2] + s[3]);
  text = kGeneral ? t : key0 < L ? sum : 0.f;
}

// The sum of the bf16 numerators of a half.
__device__ __forceinline__ float rounded_sum(const uint32_t (&w)[32]) {
  float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int e = 0; e < 32; ++e)
    fadd2(s[2 * (e & 1)], s[2 * (e & 1) + 1], __uint_as_float(w[e] << 16),
          __uint_as_float(w[e] & 0xffff0000u));
  return (s[0] + s[1]) + (s[2] + s[3]);
}

struct RowState {
  float m;        // reference
  float la, lt;   // sums over all keys, over the text keys
  float dr;       // what rounding P to bf16 added to the row's large halves
};

// One half of the rows' key tile (the whole warp): exponentials, sums and P
// against the rows' references.  When a row's sum passes kJump (its first
// keys, a term far above the reference, NaN) that row takes the half's maximum
// as its reference (at a row's first keys the whole key tile's: t_next is the
// other half's S columns), and the warp's exponentials are taken once more; the
// other rows' come out the same.
// A term that dominates its row and is not a power of two is rounded in P and
// would carry that error into O / la whole: where the row's own sum, before any
// such move, passed kBig (`big`), the caller adds to dr the difference between
// P's sum and the exact one, and O is divided by la + dr, in which it cancels.  No
// row's result depends on another row of its warp.
// Returns the factor that the row's earlier sums (and O) were rescaled by;
// `moved`, uniform: some row's is not 1.
__device__ __forceinline__ float softmax_half(const uint32_t (&a)[32], const uint32_t (&b)[32],
                                              uint32_t (&w)[32], int key0, int Nk, int L, float c,
                                              RowState& st, float& sum, bool& moved, bool& big,
                                              uint32_t t_next) {
  // uniform: all 64 keys valid and on one side of the text's end
  const bool plain = key0 + kHalf <= Nk && (key0 >= L || key0 + kHalf <= L);
  float text, f = 1.f;
  if (plain)
    exp_half<false>(a, b, w, key0, Nk, L, c, st.m, sum, text);
  else
    exp_half<true>(a, b, w, key0, Nk, L, c, st.m, sum, text);
  big = !(sum < kBig);
  moved = false;
  if (__any_sync(0xffffffffu, big)) {
    const bool over = !(sum < kJump);
    moved = __any_sync(0xffffffffu, over);
    if (moved) {
      float next = -INFINITY;
      if (t_next) {
#pragma unroll 1
        for (int k = 0; k < 2; ++k) {
          uint32_t r[32];
          tmem_ld32_wait(t_next + (uint32_t)(32 * k), r);
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if (key0 + kHalf + 32 * k + e < Nk) next = fmaxf(next, __uint_as_float(r[e]));
        }
      }
      if (over) {
        const float mx = plain ? half_max<false>(a, b, key0, Nk) : half_max<true>(a, b, key0, Nk);
        const float m = fmaxf(st.m, fmaxf(mx, next) * c);
        f = ex2(st.m - m);
        st.la *= f;
        st.lt *= f;
        st.dr *= f;
        st.m = m;
      }
      if (plain)
        exp_half<false>(a, b, w, key0, Nk, L, c, st.m, sum, text);
      else
        exp_half<true>(a, b, w, key0, Nk, L, c, st.m, sum, text);
    }
  }
  st.la += sum;
  st.lt += text;
  return f;
}

// Indices of a key tile's K and V loads in the ring: the load order is the
// order the MMAs consume them.
__device__ __forceinline__ int k_load(int g) { return 2 * g; }
__device__ __forceinline__ int v_load(int g) { return 2 * g + 1; }

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
attention_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
                    const AttnParams p) {
  using C = Cfg<D>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sQ = smem;
  uint8_t* sKV = sQ + C::kQBytes;
  uint8_t* sStage = sKV + C::kKVBytes;   // O staging, one 64-column block per tile
  Bars* bars = reinterpret_cast<Bars*>(sStage + kStageBytes);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int n_my = (p.n_units - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  if (n_my <= 0) return;   // block-uniform
  const int G = n_my * p.n_kt;   // key tiles this CTA processes (all its units)

  if (threadIdx.x == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmQ)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmK)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmV)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmO)) : "memory");
    for (int t = 0; t < kQTiles; ++t) {
      mbar_init(&bars->q_full[t], 1);
      mbar_init(&bars->q_empty[t], 1);
      mbar_init(&bars->s_full[t], 1);
      mbar_init(&bars->p_full[t][0], 4);   // the tile's 4 softmax warps
      mbar_init(&bars->p_full[t][1], 4);
      mbar_init(&bars->pv_half[t], 1);
      mbar_init(&bars->o_full[t], 1);
      mbar_init(&bars->o_empty[t], 4);
      mbar_init(&bars->turn[t], 1);
      mbar_init(&bars->drain[t], 1);
    }
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(&bars->kv_full[s], 1);
      mbar_init(&bars->kv_empty[s], kQTiles);   // one commit per issuer
    }
    bars->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_shared();
  }
  // Q, K and V may come from the kernel before this one on the stream
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (warp == 1) tmem_alloc(&bars->tmem_base, kTmemCols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = bars->tmem_base;
  volatile int* abort_flag = &bars->abort;
  if (threadIdx.x == 96) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  auto unit_coords = [&](int u, int& b, int& h, int& qp) {
    const int bh = u / p.n_qp;
    qp = u - bh * p.n_qp;
    b = bh / p.H;
    h = bh - b * p.H;
  };

  if (warp < 4) {
    // 128 x 88 + 256 x 208 = 384 x 168, what the block was launched with
    asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
    // ------------------------------------------------------ TMA producer --
    if (warp == 0) {
      bool ok = true;
      int loads = 0;                 // K and V tiles armed so far, ring position
      int q_armed = 0, q_unit = 0;   // Q tiles armed for unit q_unit
      int b, h, qp;
      auto load_q = [&](int ui, int t) {
        if (ui > 0)
          ok = mbar_wait_bounded(&bars->q_empty[t], (uint32_t)((ui - 1) & 1), abort_flag, p.status);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) return;
        q_armed = t + 1;
        q_unit = ui;
        if (elect_one()) {
          mbar_arrive_expect_tx(&bars->q_full[t], C::kTileBytes);
          for (int cb = 0; cb < C::kCB; ++cb)
            tma_load_4d(sQ + t * C::kTileBytes + cb * (kBM * 128), &tmQ, cb * 64,
                        qp * kUnitRows + t * kBM, h, b, &bars->q_full[t]);
        }
        __syncwarp();
      };
      // the ring's next load: key tile kt of the unit
      auto load_kv = [&](const CUtensorMap* map, int kt) {
        const int stage = loads % C::kStages;
        const uint32_t ph = (uint32_t)((loads / C::kStages) & 1);
        ok = mbar_wait_bounded(&bars->kv_empty[stage], ph ^ 1u, abort_flag, p.status);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) return;
        ++loads;
        if (elect_one()) {
          mbar_arrive_expect_tx(&bars->kv_full[stage], C::kTileBytes);
          for (int cb = 0; cb < C::kCB; ++cb)
            tma_load_4d(sKV + stage * C::kTileBytes + cb * (kBM * 128), map, cb * 64, kt * kBN, h, b,
                        &bars->kv_full[stage]);
        }
        __syncwarp();
      };
      for (int ui = 0; ui < n_my && ok; ++ui) {
        unit_coords((int)blockIdx.x + ui * (int)gridDim.x, b, h, qp);
        load_q(ui, 0);
        if (ok && ui > 0) load_q(ui, 1);
        if (ok) load_kv(&tmK, 0);
        if (ok && ui == 0) load_q(ui, 1);   // the first K tile ahead of it at the start
        if (ok) load_kv(&tmV, 0);
        for (int kt = 1; kt < p.n_kt && ok; ++kt) {
          load_kv(&tmK, kt);
          if (ok) load_kv(&tmV, kt);
        }
      }
      if (!ok) {
        // drain the copies still in flight before the CTA exits
        for (int t = 0; t < q_armed; ++t)
          mbar_wait_bounded(&bars->q_full[t], (uint32_t)(q_unit & 1), nullptr, p.status);
        for (int i = loads > C::kStages ? loads - C::kStages : 0; i < loads; ++i)
          mbar_wait_bounded(&bars->kv_full[i % C::kStages], (uint32_t)((i / C::kStages) & 1),
                            nullptr, p.status);
      }
    }
    // -------------------------------------------------------- MMA issuers --
    // S_t(0); then per key tile g a turn: the two halves of O_t += P_t(g) V_g
    // and S_t(g+1) behind them.  The tensor pipe runs one thread's products in
    // the order they were issued, so S_t(g+1) may overwrite P_t(g).
    if (warp == 1 || warp == 2) {
      const int t = warp - 1;
      const uint32_t q_lo = sw128_desc_lo(sQ + t * C::kTileBytes);
      const uint32_t kv_lo0 = sw128_desc_lo(sKV);
      const uint32_t v_lo0 = sw128_mn_desc_lo(sKV, kBM * 128);
      const uint32_t d_hi = sw128_desc_hi();
      const uint32_t tS = tmem + (uint32_t)(kColS + t * kBN);
      const uint32_t tO = tmem + (uint32_t)(kColO + t * D);
      bool ok = true;
      auto wait = [&](uint64_t* bar, int phase) {
        if (ok) ok = mbar_wait_bounded(bar, (uint32_t)(phase & 1), abort_flag, p.status);
      };
      int s_u = 0;   // unit of the next S
      auto issue_s = [&](int lk, bool last) {   // lk: the K tile's number in the ring
        const uint32_t k_lo = kv_lo0 + (uint32_t)(((lk % C::kStages) * C::kTileBytes) >> 4);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint32_t off = (uint32_t)(((kk >> 2) * (kBM * 128) + (kk & 3) * 32) >> 4);
            mma_ss(tS, q_lo + off, k_lo + off, d_hi, kIdescS, kk > 0 ? 1u : 0u);
          }
          mma_commit(&bars->s_full[t]);
          mma_commit(&bars->kv_empty[lk % C::kStages]);
          if (last) mma_commit(&bars->q_empty[t]);
        }
        __syncwarp();
      };
      auto pass_turn = [&]() {
        if (lane == 0) mbar_arrive(&bars->turn[t ^ 1]);
      };
      wait(&bars->kv_full[0], 0);
      wait(&bars->q_full[t], 0);
      if (t == 1) wait(&bars->turn[1], 0);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) {
        issue_s(k_load(0), p.n_kt == 1);
        pass_turn();
      }
      int v_j = 0, v_u = 0;   // key tile within the unit, and unit, of P V
      for (int g = 0; g < G && ok; ++g) {
        const int lv = v_load(g), lk = k_load(g + 1);
        const bool more = g + 1 < G, next_unit = v_j == p.n_kt - 1;
        // waited for while the other tile has its turn
        if (v_j == 0 && v_u > 0) wait(&bars->o_empty[t], v_u - 1);   // O_t of the previous unit is read
        wait(&bars->kv_full[lv % C::kStages], lv / C::kStages);
        if (more && !next_unit) wait(&bars->kv_full[lk % C::kStages], lk / C::kStages);
        wait(&bars->p_full[t][0], g);
        wait(&bars->turn[t], t == 0 ? g : g + 1);
        const uint32_t v_lo = v_lo0 + (uint32_t)(((lv % C::kStages) * C::kTileBytes) >> 4);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          if (hf == 1) wait(&bars->p_full[t][1], g);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          fence_after();
          if (elect_one()) {
#pragma unroll
            for (int k4 = 0; k4 < kHalf / 16; ++k4) {   // 16 keys: 8 P columns, 16 V rows
              const int kk = hf * (kHalf / 16) + k4;
              mma_ts(tO, tS + (uint32_t)(kk * 8), v_lo + (uint32_t)((kk * 16 * 128) >> 4), d_hi,
                     C::kIdescPV, (v_j > 0 || kk > 0) ? 1u : 0u);
            }
            if (hf == 0) {
              mma_commit(&bars->pv_half[t]);
            } else {
              mma_commit(&bars->kv_empty[lv % C::kStages]);
              if (next_unit) mma_commit(&bars->o_full[t]);
            }
          }
          __syncwarp();
        }
        if (!ok) break;
        if (more) {
          if (next_unit) {
            ++s_u;
            wait(&bars->q_full[t], s_u);
            wait(&bars->kv_full[lk % C::kStages], lk / C::kStages);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
          }
          const int s_j = next_unit ? 0 : v_j + 1;
          issue_s(lk, s_j == p.n_kt - 1);
        }
        pass_turn();
        if (next_unit) { v_j = 0; ++v_u; } else { ++v_j; }
      }
      // all issued MMAs complete before tensor memory is released
      if (elect_one()) mma_commit(&bars->drain[t]);
      __syncwarp();
      mbar_wait_bounded(&bars->drain[t], 0, nullptr, p.status);
    }
  } else {
    // --------------------------------------------- softmax and epilogue --
    asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
    const int t = (warp - 4) >> 2;
    const int quad = warp & 3;             // TMEM lane quadrant this warp may access
    const int rowt = quad * 32 + lane;     // row within the tile = TMEM lane
    const bool leader = (quad == 0 && lane == 0);
    // named barrier of the tile's 128 threads: 1 + t (literal ids, so that
    // the kernel reserves only the barriers it uses)
    auto tile_sync = [&]() { if (t == 0) bar_sync(1, 128); else bar_sync(2, 128); };
    auto tile_and = [&](bool v) { return t == 0 ? bar_and(1, 128, v) : bar_and(2, 128, v); };
    const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
    const uint32_t tS = tmem + lane_off + (uint32_t)(kColS + t * kBN);
    const uint32_t tO = tmem + lane_off + (uint32_t)(kColO + t * D);
    uint8_t* sSt = sStage + t * kStageTileBytes;
    const float c = p.c_log2;
    bool ok = true;
    int gi = 0;
    for (int ui = 0; ui < n_my; ++ui) {
      int b, h, qp;
      unit_coords((int)blockIdx.x + ui * (int)gridDim.x, b, h, qp);
      RowState st{-INFINITY, 0.f, 0.f, 0.f};
      for (int j = 0; j < p.n_kt; ++j, ++gi) {
        ok = ok && (*abort_flag == 0) &&
             mbar_wait_bounded(&bars->s_full[t], (uint32_t)(gi & 1), abort_flag, p.status);
        ok = __all_sync(0xffffffffu, ok);   // tcgen05.ld / st are warp-collective
        if (!ok) continue;
        fence_after();
        // one body for both halves: 5 KB of straight-line code that stays in
        // the instruction cache
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          uint32_t r0[32], r1[32], w[32];
          tmem_ld64_wait(tS + (uint32_t)(h * kHalf), r0, r1);
          bool moved, big;
          float sum;
          const float f = softmax_half(r0, r1, w, j * kBN + h * kHalf, p.Nk, p.L, c, st, sum, moved,
                                       big, j + h == 0 ? tS + (uint32_t)kHalf : 0u);
          if (moved && j + h > 0) {
            // O_t holds the products before this half (S_t complete: all of the
            // earlier tiles'; the first half's is waited for)
            if (h == 1) {
              ok = mbar_wait_bounded(&bars->pv_half[t], (uint32_t)(gi & 1), abort_flag, p.status);
              ok = __all_sync(0xffffffffu, ok);
              if (!ok) break;
              fence_after();
            }
            rescale_o<D>(tO, f);
          }
          // P over S columns that are in registers
          tmem_st32(tS + (uint32_t)(h * (kHalf / 2)), w);
          tmem_wait_st();
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars->p_full[t][h]);
          // behind the hand-over: nothing waits for it
          if (__any_sync(0xffffffffu, big)) {
            const float d = rounded_sum(w) - sum;
            if (big) st.dr += d;
          }
        }
      }
      // ---- epilogue: O / l -> bf16 -> swizzled staging, 64 columns at a
      // time -> TMA store
      ok = ok && (*abort_flag == 0) &&
           mbar_wait_bounded(&bars->o_full[t], (uint32_t)(ui & 1), abort_flag, p.status);
      ok = __all_sync(0xffffffffu, ok);
      const float inv = 1.f / (st.la + st.dr);
      const int row0 = qp * kUnitRows + t * kBM;
#pragma unroll 1
      for (int cb = 0; cb < C::kCB; ++cb) {
        if (ok) {
          fence_after();
#pragma unroll 1
          for (int k = 0; k < 2; ++k) {
            uint32_t r[32];
            tmem_ld32_wait(tO + (uint32_t)(64 * cb + 32 * k), r);
            uint32_t w[16];
#pragma unroll
            for (int e = 0; e < 16; ++e)
              w[e] = pack_bf16x2(__uint_as_float(r[2 * e]) * inv, __uint_as_float(r[2 * e + 1]) * inv);
            uint8_t* rowp = sSt + rowt * 128;
#pragma unroll
            for (int q = 0; q < 4; ++q)
              *reinterpret_cast<uint4*>(rowp + (((4 * k + q) ^ (rowt & 7)) << 4)) =
                  make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
          }
          fence_before();
        }
        if (cb == C::kCB - 1) {   // every O column of this unit has been read
          __syncwarp();
          if (ok && lane == 0) mbar_arrive(&bars->o_empty[t]);
        }
        fence_async_shared();
        const bool all_ok = tile_and(ok);
        if (all_ok && leader && row0 < p.Mq) {   // a tile past the end stores nothing
          tma_store_4d(&tmO, sSt, cb * 64, row0, h, b);
          bulk_commit();
          bulk_wait_read();   // the staging is rewritten by the next block
        }
        tile_sync();
      }
      const int row = row0 + rowt;
      if (ok && row < p.Mq) {
        const float ln2 = 0.69314718055994530942f;
        if (p.lse) {
          float* lp = p.lse + (((long long)b * p.H + h) * p.Mq + row) * 2;
          lp[0] = (st.m + log2f(st.la)) * ln2;
          lp[1] = st.lt > 0.f ? (st.m + log2f(st.lt)) * ln2 : -INFINITY;
        }
        if (p.A)
          head_sum_add(p.acc + (long long)b * p.rows_pad + row, p.H, st.lt / st.la, p.weight,
                       p.accumulate, p.A + (long long)b * p.Mq + row);
      }
    }
    if (leader) bulk_wait_all();
  }

  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

struct Plan {
  int n_qp, n_kt, n_units, grid;
  size_t acc_bytes;
};

Plan make_plan(int B, int H, int Mq, int Nk, int num_sms) {
  Plan pl{};
  pl.n_qp = (Mq + kUnitRows - 1) / kUnitRows;
  pl.n_kt = (Nk + kBN - 1) / kBN;
  pl.n_units = B * H * pl.n_qp;
  const int sms = num_sms > 0 ? num_sms : 1;
  pl.grid = pl.n_units < sms ? pl.n_units : sms;
  pl.acc_bytes = (sizeof(unsigned long long) * (size_t)B * pl.n_qp * kUnitRows + 255) &
                 ~static_cast<size_t>(255);
  return pl;
}

template <auto Kernel, int D>
cudaError_t smem_attrs() {
  cudaError_t e = cudaFuncSetAttribute(Kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes<D>());
  return e;
}

cudaError_t set_smem_once() {
  static int done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && __atomic_load_n(&done[dev], __ATOMIC_ACQUIRE)) return cudaSuccess;
  e = smem_attrs<attention_tc_kernel<128>, 128>();
  if (e == cudaSuccess) e = smem_attrs<attention_tc_kernel<64>, 64>();
  if (e == cudaSuccess && dev >= 0 && dev < 64) __atomic_store_n(&done[dev], 1, __ATOMIC_RELEASE);
  return e;
}

static_assert(smem_bytes<128>() <= 232448, "attention kernel shared memory above the opt-in limit");

}  // namespace

size_t attention_tc_workspace(int B, int H, int Mq) {
  return make_plan(B, H, Mq, 1, 1).acc_bytes;
}

bool attention_tc_layout_ok(const AttnArgs& a) {
  if (a.d != 64 && a.d != 128) return false;
  const void* ptrs[4] = {a.q, a.k, a.v, a.o};
  for (const void* ptr : ptrs)
    if (reinterpret_cast<uintptr_t>(ptr) & 15u) return false;
  for (int i = 0; i < 4; ++i)
    if (!strides_ok(a.B, a.H, a.str[i][0], a.str[i][1], a.str[i][2])) return false;
  return encode_fn() != nullptr;
}

cudaError_t launch_attention_tc(const AttnArgs& a, int num_sms, cudaStream_t s) {
  const Plan pl = make_plan(a.B, a.H, a.Mq, a.Nk, num_sms);
  CUtensorMap mq, mk, mv, mo;
  if (!make_map(&mq, a.q, a.B, a.H, a.Mq, a.d, a.str[0][0], a.str[0][1], a.str[0][2]) ||
      !make_map(&mk, a.k, a.B, a.H, a.Nk, a.d, a.str[1][0], a.str[1][1], a.str[1][2]) ||
      !make_map(&mv, a.v, a.B, a.H, a.Nk, a.d, a.str[2][0], a.str[2][1], a.str[2][2]) ||
      !make_map(&mo, a.o, a.B, a.H, a.Mq, a.d, a.str[3][0], a.str[3][1], a.str[3][2]))
    return cudaErrorInvalidValue;
  AttnParams p{};
  p.B = a.B; p.H = a.H; p.Mq = a.Mq; p.Nk = a.Nk; p.L = a.L;
  p.n_qp = pl.n_qp; p.n_kt = pl.n_kt; p.n_units = pl.n_units;
  p.c_log2 = a.scale * 1.4426950408889634f;
  p.weight = a.weight;
  p.accumulate = a.accumulate;
  p.A = a.A;
  p.lse = a.lse;
  p.acc = static_cast<unsigned long long*>(a.ws);
  p.rows_pad = pl.n_qp * kUnitRows;
  p.status = a.status;
  cudaError_t e = set_smem_once();
  if (e != cudaSuccess) return e;
  if (a.d == 128)
    e = launch_pdl(attention_tc_kernel<128>, dim3(pl.grid), dim3(kThreads), smem_bytes<128>(), s,
                   mq, mk, mv, mo, p);
  else
    e = launch_pdl(attention_tc_kernel<64>, dim3(pl.grid), dim3(kThreads), smem_bytes<64>(), s,
                   mq, mk, mv, mo, p);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace avits
