// Non-causal attention of the bidirectional forward (Eq. 2 runs one full pass in which
// every position attends to every position of its sequence), on the tcgen05 tensor
// cores of sm_103a.
//
// The unit of query work is a band: 32 consecutive query rows of one head.  One CTA takes up
// to eight bands of one (sequence, kv head), two tiles of four: consecutive rows of a head
// with multi-head attention, rows of the heads that share the kv head with grouped queries
// (so a step that computes 32 rows of a sequence loads its keys once for four heads of a tile,
// not once per head).  The key axis is walked in blocks of 128: S = Q K^T into TMEM per tile,
// then per row a running maximum m, P = exp2(S * log2(e)/sqrt(hd) - m) with the row sum l kept
// in fp32, P written to shared memory in fp16 (11 significant bits; P <= 2^8), and O += P V in
// TMEM with V^T held in fp16 (the bf16 values of v, which fp16 holds exactly).  m moves only
// when a block's maximum exceeds it by more than 8 (P stays below 2^8); l and O are then scaled
// by the same factor, so O / l is unchanged.  m is held and exchanged in fp32: P passes 2^8 by as
// much as m misses the maximum (an m rounded to bf16 gave infinities from scores of about 1400
// on).  O / l leaves through TMA.
//
// What bounds it now is shared memory: per key block of two tiles the products read 256 KB of
// operands, P is written (64 KB) and the block arrives (64 KB), 3072 cycles at 128 bytes a cycle
// against 3100 measured and 2048 of tensor time.  Before that the issue of the MMAs was the
// bound (one thread of a diverged warp: 4450 cycles, whatever the softmax did).  Sixteen warps
// share the softmax: two per band, each on one 64-column half of a block (64 scores a thread
// leave room for all of them in registers).  S is free for the next block's product as soon as
// its scores and the halves' maxima have been read.  Two tiles per CTA keep four such warps on
// every scheduler and load each key block once for 256 rows.
// Measured against one tile per CTA with eight softmax warps (kernel, us): 8 x 1536 positions,
// 32 heads of 128: 430 -> 265 (1166 TFLOP/s); 4 x 1000, 28 q / 4 kv heads: 81 -> 52; 1 x 512: 9.3
// -> 9.6; 32 query rows of each of 16 x 896 (28 / 4 heads): 55 -> 13; 32 rows of 1 x 1536: 18.9
// -> 9.8.
//
// A launch has at most one CTA per SM (each takes nearly all of its shared memory), which walk
// the units of the rows there are: a grid laid out for the most rows left empty CTAs that each
// waited for a whole SM (the current blocks of 8 x 1536 positions, 256 units of one band in 1536
// CTAs: 79 us a layer, walked 44).  Consecutive units are the kv heads of one sequence, then its
// next rows, so that the keys and values in use stay in L2.  With a CTA for each unit 8 x 1536
// took 281 us and 4 x 1000 55; one unit a CTA of twelve key blocks pays for the walk (544 rows of
// 1 x 1536: 24.7 -> 25.4).
//
// Where the units of a launch leave SMs idle the key axis is split over the S CTAs of a
// cluster: each keeps (m, l, O) of its blocks, and after one cluster barrier every CTA
// combines 1 / S of the rows, reading the S parts through distributed shared memory (in rank
// order, so bit-reproducible).  Whether a launch splits, and takes four or eight bands per CTA,
// follows from the rows that the row plan gives it (attn_cost); without the split a cluster's
// CTAs are independent.
//
// Roles (576 threads): warp 0 TMA producer (a unit's Q, then K / V^T blocks through a ring in the
// order the MMAs consume them; one elected lane issues); warp 1 allocates TMEM and issues the
// MMAs (a second issuer, a warp per tile, gained nothing); warps 2..17 run the softmax and the
// epilogue (TMEM lane quarter = band of the tile).  V enters as V^T (a K-major operand, kv
// contiguous, fp16), written by the QKV GEMM's epilogue or by v_transpose_kernel from the q|k|v
// buffer.
// Every wait is bounded (DERR_WAIT_TIMEOUT).
#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace dcl {
namespace {

// The value of lane 0, which the compiler then knows to be the whole warp's (uniform registers, no
// divergence in what depends on it).
__device__ __forceinline__ int warp_uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }

constexpr int AT_SOFTMAX = 8;  // softmax warps of a tile
constexpr int AT_THREADS = 64 + 2 * 32 * AT_SOFTMAX;
constexpr int AT_BOX = 128 * 128;  // one 128-row x 128-byte swizzle box

// A unit of query work: `live` bands (0: none is left) of kv head g of sequence b, each 32 rows of a
// query head from row[i] of q and of the output, column col[i]; rows from `end` on are not the
// sequence's.
struct AttnUnit {
  int g, b, end, live;
  int row[8], col[8];
};
// How a launch's rows are cut: bands per unit; whether the keys of a unit are split over the
// cluster, and this CTA's key blocks [jb, jb + n).  dead: a wait of this CTA has run out.  b0,
// before: the 32 sequences that the last unit was found in, and the units of those before them.
struct AttnLaunch {
  int bands, split, jb, n, dead, b0, before;
};

template <int HD>
struct AttnCfg {
  static constexpr int KB = HD / 64;                // 64-wide boxes along hd
  static constexpr int Q_BYTES = 128 * HD * 2;      // a tile of Q [128][HD]
  static constexpr int STAGES = HD == 128 ? 3 : 6;
  static constexpr int STAGE_BYTES = 128 * HD * 2;  // K block [128][HD] or V^T block [HD][128]
  static constexpr int VBOX = HD * 128;             // one V^T box: [HD rows][64 kv]
  static constexpr int P_BYTES = 2 * AT_BOX;        // a tile of P (fp16) [128][128]
  static constexpr int BARS = 512;                  // barriers, then two units and how they are cut
  static constexpr int DATA = 2 * Q_BYTES + STAGES * STAGE_BYTES + 2 * P_BYTES;
  static constexpr int RED = 2 * 2 * 128 * 4;       // row maxima of the halves [tile][half][row]
  // (no slack for the 1024-byte alignment, which the declaration asks for and the kernel checks:
  // 2 x 1 KB of fp32 maxima do not fit beside it)
  static constexpr size_t SMEM = (size_t)DATA + RED + BARS;
  static constexpr int BAR0 = DATA + RED, NBARS = 1 + 2 * STAGES + 8 + 1;
  static constexpr int HOLDER = BAR0 + 8 * NBARS, UNITS = HOLDER + 8, LAUNCH = UNITS + 2 * sizeof(AttnUnit);
  static_assert(LAUNCH + sizeof(AttnLaunch) <= SMEM, "barrier area");
  static constexpr uint32_t TMEM_COLS = 512;        // S of two tiles (2 x 128), O of two (2 x HD)
  // a split's parts: O rows in fp32 (padded by 16 bytes), then {m, l} of every row
  static constexpr int O_PITCH = HD * 4 + 16;
  static constexpr int ML = 256 * O_PITCH;
  static_assert(ML + 256 * 8 <= DATA, "the parts take the place of the operands");
  static_assert(SMEM <= 232448, "shared memory per CTA");
};

// Units (CTAs' worth of bands, four or eight) of a sequence with `rows` query rows.
__host__ __device__ inline int attn_units(int rows, int rep, int bands) {
  return (rep * ((rows + 31) / 32) + bands - 1) >> (bands > 4 ? 3 : 2);
}
// What `units` units of `bands` bands over nb key blocks take with the key axis split S ways, in
// tenths of a key block of two tiles: rounds of CTAs, each its blocks (one tile takes 6/10 of
// two), its start and end (2 blocks), and with a split the combination (2 blocks).
// (per_sm: 1 / SMs.  Divisions are slow and stand between a kernel's start and its first load.)
__host__ __device__ inline int attn_cost(int units, int bands, int nb, int S, float per_sm) {
  const int rounds = (int)ceilf((float)(units * S) * per_sm - 1e-3f);
  return rounds * ((nb + S - 1) / S * (bands > 4 ? 10 : 6) + (S > 1 ? 20 : 0) + 20);
}

// vt[(b*G + g)*hd + d][t] = v of token t, kv head g, component d (row pitch Tp, zero pad),
// in fp16 (the bf16 values, held exactly).  A block moves a 64-token x 64-channel tile
// with 16-byte loads and stores.
__global__ void __launch_bounds__(256) v_transpose_kernel(const __nv_bfloat16* __restrict__ qkv,
                                                          __half* __restrict__ vt, int T, int Tp, int cols,
                                                          int v0, int ghd) {
  __shared__ __half tile[64][72];  // [channel][token], rows padded by 16 bytes
  pdl_wait();
  pdl_launch_dependents();
  const int t0 = blockIdx.x * 64, c0 = blockIdx.y * 64, b = blockIdx.z;
  for (int i = threadIdx.x; i < 64 * 8; i += 256) {
    const int r = i >> 3, cv = (i & 7) * 8;  // token row, first channel of the vector
    const int t = t0 + r;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (t < T && c0 + cv < ghd)
      v = *reinterpret_cast<const uint4*>(qkv + ((size_t)b * T + t) * cols + v0 + c0 + cv);
    const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(&v);
#pragma unroll
    for (int k = 0; k < 8; ++k) tile[cv + k][r] = __float2half_rn(__bfloat162float(e[k]));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 64 * 8; i += 256) {
    const int c = i >> 3, tv = (i & 7) * 8;  // channel row, first token of the vector
    if (c0 + c < ghd && t0 + tv < Tp)
      *reinterpret_cast<uint4*>(vt + ((size_t)b * ghd + c0 + c) * Tp + t0 + tv) =
          *reinterpret_cast<const uint4*>(&tile[c][tv]);
  }
}

// The MMA issuer of a unit (warp 1; the whole warp, one lane issues).  Its operands are made known as
// the warp's: inside the loop over the units the compiler did not see it, and the issue of a block
// of two tiles took 2260 cycles instead of 2150 (2048 of tensor time).
template <int HD>
__device__ __forceinline__ void attn_mma(uint32_t base, uint32_t tmem, int ntiles, int n, volatile int* abort_flag, int* err) {
  using C = AttnCfg<HD>;
  base = (uint32_t)warp_uniform((int)base);
  tmem = (uint32_t)warp_uniform((int)tmem);
  ntiles = warp_uniform(ntiles);
  n = warp_uniform(n);
  const uint32_t sQ = base, sKV = sQ + 2 * C::Q_BYTES, sP = sKV + C::STAGES * C::STAGE_BYTES;
  const uint32_t q_full = base + C::BAR0, kv_full0 = q_full + 8, kv_empty0 = kv_full0 + 8 * C::STAGES;
  const uint32_t s_full0 = kv_empty0 + 8 * C::STAGES, s_empty0 = s_full0 + 16, p_full0 = s_empty0 + 16;
  const uint32_t p_empty0 = p_full0 + 16, drain = p_empty0 + 16;
  constexpr uint32_t idesc_s = make_idesc(128, 128);
  constexpr uint32_t idesc_o = make_idesc_f16(128, HD);  // fp16 P and V
  const bool leader = elect_one();
  auto wait = [&](uint32_t bar, uint32_t parity) {
    return (bool)__all_sync(0xffffffffu, mbar_wait_inline(bar, parity, abort_flag));
  };
  bool ok = wait(q_full, 0);
  int stage = 0;
  uint32_t phase = 0;
  auto next_stage = [&]() {
    if (++stage == C::STAGES) {
      stage = 0;
      phase ^= 1u;
    }
  };
  auto issue_s = [&](int j) -> bool {  // S = Q K_j^T of both tiles
    if (!wait(kv_full0 + 8 * stage, phase)) return false;
    const uint64_t dk = sw128_desc(sKV + stage * C::STAGE_BYTES);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      if (t >= ntiles) break;
      if (!wait(s_empty0 + 8 * t, ((uint32_t)j & 1u) ^ 1u)) return false;
      tc_fence_after();
      const uint64_t dq = sw128_desc(sQ + t * C::Q_BYTES);
      if (leader) {
#pragma unroll
        for (int k = 0; k < HD / 16; ++k)
          umma_bf16(tmem + 128u * t, dq + (k >> 2) * (AT_BOX >> 4) + 2 * (k & 3), dk + (k >> 2) * (AT_BOX >> 4) + 2 * (k & 3),
                    idesc_s, k > 0 ? 1u : 0u);
        umma_commit(s_full0 + 8 * t);
        if (t + 1 == ntiles) umma_commit(kv_empty0 + 8 * stage);
      }
      __syncwarp();
    }
    next_stage();
    return true;
  };
  auto issue_pv = [&](int j) -> bool {  // O += P_j V_j of both tiles (fp16 operands)
    if (!wait(kv_full0 + 8 * stage, phase)) return false;
    const uint64_t dv = sw128_desc(sKV + stage * C::STAGE_BYTES);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      if (t >= ntiles) break;
      if (!wait(p_full0 + 8 * t, (uint32_t)j & 1u)) return false;
      tc_fence_after();
      const uint64_t dp = sw128_desc(sP + t * C::P_BYTES);
      if (leader) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
          umma_bf16(tmem + 256u + (uint32_t)(HD * t), dp + (k >> 2) * (AT_BOX >> 4) + 2 * (k & 3),
                    dv + (k >> 2) * (C::VBOX >> 4) + 2 * (k & 3), idesc_o, (j > 0 || k > 0) ? 1u : 0u);
        umma_commit(p_empty0 + 8 * t);
        if (t + 1 == ntiles) umma_commit(kv_empty0 + 8 * stage);
      }
      __syncwarp();
    }
    next_stage();
    return true;
  };
  if (ok) ok = issue_s(0);
  for (int j = 0; ok && j < n; ++j) {  // S_{j+1} (its buffer frees early in the softmax of j) before P V of j
    if (j + 1 < n) ok = issue_s(j + 1);
    if (ok) ok = issue_pv(j);
  }
  if (!ok) {
    *abort_flag = 1;
    if (leader) report_error(err, DERR_WAIT_TIMEOUT);
  }
  if (leader) umma_commit(drain);  // every MMA issued here completes before the unit's end
  __syncwarp();
  volatile int no_abort = 0;
  mbar_wait(drain, 0, &no_abort);
}

template <int HD>
__global__ void __launch_bounds__(AT_THREADS, 1)
    attn_tc_kernel(const __grid_constant__ CUtensorMap tq, const __grid_constant__ CUtensorMap tk,
                   const __grid_constant__ CUtensorMap tv, const __grid_constant__ CUtensorMap to,
                   __nv_bfloat16* __restrict__ out, int B, int T, int H, int G, int rep, int kcol0,
                   const int* __restrict__ seq_off, const int* __restrict__ seq_len, int q_rows, int mode, int bands,
                   float per_sm, int* err) {
  using C = AttnCfg<HD>;
  extern __shared__ __align__(1024) uint8_t smem[];
  // (opaque to the compiler: with a known constant in every address it spills, 3 % of the time)
  uint32_t base = smem_u32(smem);
  asm volatile("" : "+r"(base));
  if (base & 1023u) {  // (the swizzled operands need it; uniform over the grid)
    if (threadIdx.x == 0) report_error(err, DERR_BAD_SHAPE);
    return;
  }
  const uint32_t sQ = base;                                // per tile: KB boxes
  const uint32_t sKV = sQ + 2 * C::Q_BYTES;
  const uint32_t sP = sKV + C::STAGES * C::STAGE_BYTES;    // per tile: two 64-key boxes of P
  const uint32_t red = base + C::DATA;                     // the halves' row maxima
  const uint32_t q_full = base + C::BAR0;
  const uint32_t kv_full0 = q_full + 8;                    // + 8 s
  const uint32_t kv_empty0 = kv_full0 + 8 * C::STAGES;     // + 8 s
  const uint32_t s_full0 = kv_empty0 + 8 * C::STAGES;      // + 8 tile
  const uint32_t s_empty0 = s_full0 + 16;
  const uint32_t p_full0 = s_empty0 + 16;
  const uint32_t p_empty0 = p_full0 + 16;
  const uint32_t drain = p_empty0 + 16;
  volatile uint32_t* holder_ptr = reinterpret_cast<volatile uint32_t*>(smem + C::HOLDER);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::HOLDER + 4);
  AttnUnit* units = reinterpret_cast<AttnUnit*>(smem + C::UNITS);  // this turn's and the next
  AttnLaunch& launch = *reinterpret_cast<AttnLaunch*>(smem + C::LAUNCH);

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // (warp-uniform)
  auto init_barriers = [&]() {  // (one thread)
    mbar_init(q_full, 1);
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(kv_full0 + 8 * s, 1);
      mbar_init(kv_empty0 + 8 * s, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(s_full0 + 8 * i, 1);
      mbar_init(s_empty0 + 8 * i, AT_SOFTMAX);  // the tile's softmax warps
      mbar_init(p_full0 + 8 * i, AT_SOFTMAX);
      mbar_init(p_empty0 + 8 * i, 1);
    }
    mbar_init(drain, 1);
    fence_mbar_init();
  };

  // Warp 0 plans: turn `it` takes unit w of the launch, unit r = w / G of the sequences' rows.
  auto plan = [&](int it, int w, int r, bool tables) {
    const int cut = launch.bands;
    int b = 0, z = 0, off = 0, len = 0;
    if (!tables) {  // the last q_rows positions of every sequence
      const int per = attn_units(q_rows, rep, cut);
      b = r / per;
      z = r - b * per;
      if (b < B) {
        off = b * T + T - q_rows;
        len = q_rows;
      }
    } else {  // rows [seq_off, seq_off + seq_len) of q and of the output
      int b0 = launch.b0, before = launch.before;  // (a CTA's units come in order)
      for (; b0 < B; b0 += 32) {
        const bool is = b0 + lane < B;
        const int n = is ? seq_len[b0 + lane] : 0, o = is ? seq_off[b0 + lane] : 0, own = attn_units(n, rep, cut);
        int upto = own;
#pragma unroll 1
        for (int d = 1; d < 32 && d < B; d <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, upto, d);
          if (lane >= d) upto += t;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, r < before + upto);
        if (hit) {
          const int l = __ffs(hit) - 1;
          b = b0 + l;
          z = r - before - __shfl_sync(0xffffffffu, upto - own, l);
          len = __shfl_sync(0xffffffffu, n, l);
          off = __shfl_sync(0xffffffffu, o, l);
          break;
        }
        before += __shfl_sync(0xffffffffu, upto, 31);
      }
      __syncwarp();
      if (lane == 0) {
        launch.b0 = b0;
        launch.before = before;
      }
    }
    AttnUnit& u = units[it & 1];
    const int nch = (len + 31) / 32, g = w - r * G;
    if (lane < 8 && len > 0) {  // band i: rows 32 (i % nch) .. of the kv head's query head i / nch
      const int band = z * cut + lane;
      int h = (int)__fdividef((float)band, (float)nch);
      h -= h * nch > band;
      h += (h + 1) * nch <= band;
      u.row[lane] = off + 32 * (band - h * nch);
      u.col[lane] = (g * rep + h) * HD;
    }
    if (lane == 0) {
      u.g = g;
      u.b = b;
      u.end = off + len;
      u.live = len > 0 ? min(cut, rep * nch - z * cut) : 0;
    }
  };

  // set-up first (it reads nothing that earlier kernels write), so that under programmatic
  // dependent launch it overlaps the tail of the kernel before
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    init_barriers();
    prefetch_tmap(&tq);
    prefetch_tmap(&tk);
    prefetch_tmap(&tv);
    prefetch_tmap(&to);
  }
  if (warp == 1) tmem_alloc(base + C::HOLDER, C::TMEM_COLS);
  // warp 0: how the launch's rows are cut, and the first unit, as far as they do not depend on the row plan
  const int S = (int)cluster_size();
  if (warp == 0) {
    const int rank = (int)cluster_rank(), nb = (T + 127) / 128;
    const int sh = 31 - __clz(S), w1 = (int)blockIdx.x, wS = w1 >> sh, r1 = w1 / G, rS = wS / G;  // whole, split
    auto set = [&](int cut, bool keys) {
      if (lane == 0) {
        launch.bands = cut;
        launch.split = keys;
        launch.jb = keys ? rank * nb >> sh : 0;
        launch.n = (keys ? (rank + 1) * nb >> sh : nb) - launch.jb;
        launch.dead = launch.b0 = launch.before = 0;
      }
      __syncwarp();
    };
    bool keys = mode == ATTN_SPLIT;
    if (mode != ATTN_BY_ROWS) {
      set(bands, keys);
      plan(0, keys ? wS : w1, keys ? rS : r1, false);
    }
    pdl_wait();  // the previous kernels of the step (the row plan among them) have completed
    if (mode != ATTN_BY_ROWS) {  // with tables: was that so, every sequence with all its rows?
      bool so = true;
      for (int i = lane; seq_len && i < B; i += 32) so = so && seq_len[i] == q_rows && seq_off[i] == i * T + T - q_rows;
      if (!__all_sync(0xffffffffu, so)) plan(0, keys ? wS : w1, keys ? rS : r1, true);
    } else {  // the cheapest of whole or split units of eight or four bands
      int total[2] = {0, 0};     // of eight, of four
      for (int i = lane; i < B; i += 32)
#pragma unroll
        for (int k = 0; k < 2; ++k) total[k] += attn_units(seq_len[i], rep, 8 >> k);
      int best = 0, cut = 8;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int n = (int)__reduce_add_sync(0xffffffffu, (unsigned)total[k]) * G;
        const int whole = attn_cost(n, 8 >> k, nb, 1, per_sm), parts = attn_cost(n, 8 >> k, nb, S, per_sm);
        if (k == 0 || whole < best) best = whole, cut = 8 >> k, keys = false;
        if (S > 1 && parts < best) best = parts, cut = 8 >> k, keys = true;
      }
      set(cut, keys);
      plan(0, keys ? wS : w1, keys ? rS : r1, true);
    }
  } else {
    pdl_wait();
  }
  pdl_launch_dependents();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *holder_ptr;
  const bool split = warp_uniform(launch.split) != 0;
  const int jb = warp_uniform(launch.jb), n = warp_uniform(launch.n);  // its key blocks of each unit

#pragma unroll 1
  for (int it = 0;; ++it) {
    const AttnUnit& u = units[it & 1];
    const int live = warp_uniform(u.live), ntiles = (live + 3) / 4;
    if (live == 0) break;  // (uniform over the CTA, and if split over the cluster)
    const int g = warp_uniform(u.g), b = warp_uniform(u.b);
    const bool dead = warp_uniform(launch.dead) != 0;
    auto plan_next = [&]() {
      const int i = (int)blockIdx.x + (it + 1) * (int)gridDim.x, w = split ? i >> (31 - __clz(S)) : i;
      plan(it + 1, w, w / G, seq_len != nullptr);
    };
    if (dead) {  // (only the cluster's barriers remain, for the CTAs that may still be at work)
      if (warp == 0) plan_next();
    } else if (warp == 0) {
      // ------------------------------------------------ TMA producer (the whole warp, one lane issues)
      const bool leader = elect_one();
      bool ok = true;
      int stage = 0;
      uint32_t phase = 0;
      if (leader) mbar_arrive_expect_tx(q_full, live * 32 * HD * 2);
      __syncwarp();
      if (lane < live) {
        const int row = u.row[lane], col = u.col[lane];
        const uint32_t dst = sQ + (lane >> 2) * C::Q_BYTES + (lane & 3) * (32 * 128);
        for (int bx = 0; bx < C::KB; ++bx) tma_load_2d(dst + bx * AT_BOX, &tq, col + bx * 64, row, q_full);
      }
      __syncwarp();
      // consumption order: K_0, then per block K_{j+1}, V_j
      for (int i = 0; i < 2 * n; ++i) {
        const bool is_v = i == 2 * n - 1 || (i > 0 && (i & 1) == 0);
        const int j = jb + (is_v ? (i - 1) >> 1 : (i + 1) >> 1);
        if (!__all_sync(0xffffffffu, mbar_wait_inline(kv_empty0 + 8 * stage, phase ^ 1u, abort_flag))) {
          ok = false;
          break;
        }
        if (leader) {
          const uint32_t dst = sKV + stage * C::STAGE_BYTES, bar = kv_full0 + 8 * stage;
          mbar_arrive_expect_tx(bar, C::STAGE_BYTES);
          if (!is_v) {
            for (int bx = 0; bx < C::KB; ++bx)
              tma_load_3d(dst + bx * AT_BOX, &tk, kcol0 + g * HD + bx * 64, j * 128, b, bar);
          } else {
            for (int bx = 0; bx < 2; ++bx) tma_load_3d(dst + bx * C::VBOX, &tv, j * 128 + bx * 64, 0, b * G + g, bar);
          }
        }
        __syncwarp();
        if (++stage == C::STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
      plan_next();
      // (the ring is left empty: the barriers start anew with the next unit)
      for (int s = 0; ok && s < C::STAGES && s < 2 * n; ++s)
        ok = __all_sync(0xffffffffu, mbar_wait_inline(kv_empty0 + 8 * s, (uint32_t)((2 * n - 1 - s) / C::STAGES) & 1u, abort_flag));
      if (!ok) {
        *abort_flag = 1;
        if (leader) report_error(err, DERR_WAIT_TIMEOUT);
      }
    } else if (warp == 1) {
      attn_mma<HD>(base, tmem, ntiles, n, abort_flag, err);
    } else {
      // ------------------------------------------------ softmax + epilogue (warps 2..17)
      const int w = warp - 2, tile = w / AT_SOFTMAX, hs = (w >> 2) & 1;  // hs: which 64 columns of a block
      const int q = warp & 3;                                            // TMEM lane quarter = band of the tile
      const int r = q * 32 + lane;                                       // query row within the tile
      const bool work = 4 * tile + q < live;
      const uint32_t lane_off = (uint32_t)(q * 32) << 16;
      const uint32_t ts = tmem + lane_off + 128u * tile + 64u * hs;
      const uint32_t to_col = tmem + lane_off + 256u + (uint32_t)(HD * tile);
      const uint32_t sPt = sP + tile * C::P_BYTES;
      const uint32_t s_full = s_full0 + 8 * tile, s_empty = s_empty0 + 8 * tile, p_full = p_full0 + 8 * tile,
                     p_empty = p_empty0 + 8 * tile;
      const uint32_t top = red + (uint32_t)(4 * ((tile * 2 + hs) * 128 + r));  // (the other half's: ^ 512)
      auto band_bar = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1u + 4u * tile + q) : "memory"); };  // the band's two warps
      constexpr int OH = HD / 2;  // O columns of this warp: [hs * OH, + OH)
      const float scale2 = kLog2e * rsqrtf((float)HD);
      bool ok = true;
      float m = -INFINITY, l = 0.f;
      auto wait = [&](uint32_t bar, int j) {
        return (bool)__all_sync(0xffffffffu, mbar_wait_inline(bar, (uint32_t)j & 1u, abort_flag));
      };
      if (!work && tile < ntiles) {  // a band past the unit's last: its warps only let the others go on
        for (int j = 0; ok && j < n; ++j) {
          ok = wait(s_full, j);
          if (lane == 0 && ok) mbar_arrive(s_empty);
          if (ok && j > 0) ok = wait(p_empty, j - 1);
          __syncwarp();
          if (lane == 0 && ok) mbar_arrive(p_full);
        }
      }
      // (one branch: scores that are loaded in one branch and used in another count as held from unit
      // to unit, 600 bytes of spills.  No early exit: both warps of a band meet at every barrier)
      for (int j = 0; work && j < n; ++j) {
        if (ok) ok = wait(s_full, j);
        if (!ok) {
          band_bar();
          continue;
        }
        uint32_t v[2][32];
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < 2; ++c) tmem_ld32(ts + 32u * c, v[c]);
        tmem_ld_wait();
        tc_fence_before();
        const int valid = T - (jb + j) * 128 - 64 * hs;  // live columns of the half block
        if (valid < 64) {
          asm volatile("" ::: "memory");  // (a branch: not 64 selects in every block)
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (32 * c + e >= valid) v[c][e] = __float_as_uint(-INFINITY);
        }
        // four independent three-input maximum chains over the 64 columns
        float mx[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const uint32_t* vw = &v[t >> 1][(t & 1) * 16];
          float acc = f32(vw[0]);
#pragma unroll
          for (int e = 1; e < 15; e += 2) acc = max3f(acc, f32(vw[e]), f32(vw[e + 1]));
          mx[t] = fmaxf(acc, f32(vw[15]));
        }
        const float mm = max3f(mx[0], mx[1], fmaxf(mx[2], mx[3])) * scale2;
        // the halves agree on the block's maximum
        st_shared_f32(top, mm);
        band_bar();
        const float mb = fmaxf(mm, ld_shared_f32(top ^ 512u));
        __syncwarp();
        if (lane == 0) mbar_arrive(s_empty);  // scores and maxima read: the next block's may be written
        const bool raise = mb > m + 8.f;      // always at the first block (m = -inf)
        const bool rescale = j > 0 && __any_sync(0xffffffffu, raise);
        float f = 1.f;
        if (raise) {
          f = ex2_approx(m - mb);
          m = mb;
        }
        // P V of the block before has read this tile's P (and its O is complete)
        if (j > 0) ok = wait(p_empty, j - 1);
        if (!ok) continue;
        if (rescale) {  // warp-uniform, rare: in small pieces beside the scores
          tc_fence_after();
#pragma unroll 1
          for (int c = hs * OH; c < (hs + 1) * OH; c += 8) {
            uint32_t ov[8];
            tmem_ld8(to_col + (uint32_t)c, ov);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 8; ++e) ov[e] = __float_as_uint(f32(ov[e]) * f);
            tmem_st8(to_col + (uint32_t)c, ov);
          }
          tmem_st_wait();
          tc_fence_before();
        }
        // the half block's sum in four packed partial sums (fixed order)
        unsigned long long ls[4] = {0ull, 0ull, 0ull, 0ull};
        const unsigned long long sc2 = pk2(scale2, scale2), nm2 = pk2(-m, -m);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          uint32_t pk[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int i = 8 * (k & 3) + 2 * e;
            float y0, y1;
            upk2(ffma2(pk2(f32(v[k >> 2][i]), f32(v[k >> 2][i + 1])), sc2, nm2), y0, y1);
            const float p0 = ex2_approx(y0), p1 = ex2_approx(y1);
            ls[e] = fadd2(ls[e], pk2(p0, p1));
            pk[e] = pack_f16x2(p0, p1);  // round to nearest even: 2^-12 relative
          }
          st_shared_v4(sPt + (uint32_t)hs * AT_BOX + swz(r, k), pk[0], pk[1], pk[2], pk[3]);
        }
        float a0, a1;
        upk2(fadd2(fadd2(ls[0], ls[1]), fadd2(ls[2], ls[3])), a0, a1);
        l = l * (j > 0 ? f : 1.f) + (a0 + a1);
        tc_fence_before();
        fence_proxy_async_smem();  // P is read by the tensor cores (async proxy)
        __syncwarp();
        if (lane == 0) mbar_arrive(p_full);
      }
      if (ok && tile < ntiles) ok = wait(p_empty, n - 1);
      tc_fence_after();
      if (work) {  // the row sum, half 0 + half 1 (through the tile's Q, which every product has read)
        const uint32_t sums = sQ + (uint32_t)(tile * C::Q_BYTES + 4 * r);
        if (ok) st_shared_f32(sums + 512u * hs, l);
        band_bar();
        if (ok) l = ld_shared_f32(sums) + ld_shared_f32(sums + 512u);
      }
      if (split) {
        // every tile's operands are done with: this CTA's part takes their place
        asm volatile("bar.sync 9, %0;" ::"n"(64 * AT_SOFTMAX) : "memory");
        if (ok && work) {
          const uint32_t row = (uint32_t)(128 * tile + r), at = base + row * C::O_PITCH;
#pragma unroll 1
          for (int c = hs * OH; c < (hs + 1) * OH; c += 32) {
            uint32_t v[32];
            tmem_ld32(to_col + (uint32_t)c, v);
            tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 8; ++k)
              st_shared_v4(at + (uint32_t)(c * 4 + 16 * k), v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
          }
          if (hs == 0) {
            st_shared_f32(base + C::ML + 8 * row, m);
            st_shared_f32(base + C::ML + 8 * row + 4, l);
          }
        }
      } else if (ok && work) {
        // epilogue: O / l -> bf16 -> TMA store, each warp one 64-column box of its band (staged in
        // the tile's P, free once every P V MMA has completed)
        const float inv = 1.0f / l;
        const int row0 = u.row[4 * tile + q], col0 = u.col[4 * tile + q];
#pragma unroll 1
        for (int c = 64 * hs; c < HD; c += 128) {
          const uint32_t bx = sPt + (uint32_t)((q * C::KB + (c >> 6)) * (32 * 128));
#pragma unroll 1
          for (int hh = 0; hh < 2; ++hh) {
            uint32_t v[32];
            tmem_ld32(to_col + (uint32_t)(c + 32 * hh), v);
            tmem_ld_wait();
            float o[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = f32(v[e]) * inv;
#pragma unroll
            for (int k = 0; k < 4; ++k)
              st_shared_v4(bx + swz(lane, 4 * hh + k), pack_bf16x2(o[8 * k], o[8 * k + 1]), pack_bf16x2(o[8 * k + 2], o[8 * k + 3]),
                           pack_bf16x2(o[8 * k + 4], o[8 * k + 5]), pack_bf16x2(o[8 * k + 6], o[8 * k + 7]));
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            if (seq_off)
              tma_store_2d(&to, bx, col0 + c, row0);
            else
              tma_store_3d(&to, bx, col0 + c, row0 - b * T, b);
          }
        }
        if (lane == 0) {
          bulk_commit();
          bulk_wait_read<0>();  // the staging boxes were read (the writes complete with the grid)
        }
        __syncwarp();
      }
      if (!ok) {
        *abort_flag = 1;
        report_error(err, DERR_WAIT_TIMEOUT);
      }
      fence_proxy_async_smem();  // what was written over Q, P and the ring, before the next unit's copies
    }

    tc_fence_before();
    const bool gone = warp_uniform(__syncthreads_or(*abort_flag)) != 0;
    tc_fence_after();
    if (split) {
      if (gone && threadIdx.x == 0) launch.dead = 1;
      __syncwarp();
      cluster_sync();  // every CTA of the cluster has its part in shared memory
      if (warp > 1 && !gone) {
        const int rank = (int)cluster_rank(), end = u.end;
        // this CTA's share of the rows, four columns a thread
        const int rows = 32 * live, i1 = (rank + 1) * rows / S * (HD / 4);
        for (int i = rank * rows / S * (HD / 4) + (int)threadIdx.x - 64; i < i1; i += 64 * AT_SOFTMAX) {
          const int row = i / (HD / 4), c = 4 * (i % (HD / 4));
          const int at = u.row[row >> 5] + (row & 31);  // row of the output
          float mx = -INFINITY, ms[8], ls[8];
          float4 o[8];
#pragma unroll
          for (int s = 0; s < 8; ++s) {
            ms[s] = ls[s] = 0.f;
            o[s] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (s < S) {
              const uint32_t from = map_cluster(base, s);
              const float2 ml = ld_cluster_v2(from + C::ML + 8 * row);
              o[s] = ld_cluster_v4(from + row * C::O_PITCH + 4 * c);
              ms[s] = ml.x;
              ls[s] = ml.y;
              mx = fmaxf(mx, ml.x);
            }
          }
          float l = 0.f;
          float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int s = 0; s < 8; ++s)
            if (s < S) {
              const float f = ex2_approx(ms[s] - mx);
              l += ls[s] * f;
              a.x += o[s].x * f;
              a.y += o[s].y * f;
              a.z += o[s].z * f;
              a.w += o[s].w * f;
            }
          if (at < end) {
            const float inv = 1.0f / l;
            *reinterpret_cast<uint2*>(out + (size_t)at * H * HD + u.col[row >> 5] + c) =
                make_uint2(pack_bf16x2(a.x * inv, a.y * inv), pack_bf16x2(a.z * inv, a.w * inv));
          }
        }
      }
      __syncwarp();
      cluster_sync_relaxed();  // no CTA goes on while another may read its part
    } else if (gone) {
      break;
    }
    if (!gone && warp_uniform(units[(it + 1) & 1].live) != 0) {  // the next unit starts from fresh barriers
      if (threadIdx.x == 0) {
        for (int i = 0; i < C::NBARS; ++i) mbar_inval(q_full + 8 * i);
        init_barriers();
      }
      __syncthreads();
    }
  }

  if (*abort_flag) abort_grace();  // (copies may be in flight)
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, C::TMEM_COLS);
  }
}

// The launch's cluster size, its clusters, bands per CTA and whether the kernel decides on the
// last and on the split.
struct AttnShape {
  int S, bands, mode;
  long clusters;
};

AttnShape attn_shape(const AttnPlan& p, const AttnRows& r) {
  const int nb = (p.T + 127) / 128, rep = p.H / p.G;
  AttnShape a{1, 8, ATTN_WHOLE, 0};
  if (r.exact) {  // every sequence has r.most rows: the cheapest choice, made here
    int best = 0;
    for (int bands = 8; bands >= 4; bands -= 4) {
      const long units = (long)p.G * p.batch * attn_units(r.most, rep, bands);
      for (int S = 1; S <= 8 && S <= nb; S *= 2) {
        const int c = attn_cost((int)units, bands, nb, S, 1.0f / (float)p.sms);
        if (!a.clusters || c < best) best = c, a = {S, bands, S > 1 ? ATTN_SPLIT : ATTN_WHOLE, units};
      }
    }
  } else {
    // the rows are the row plan's.  Clusters as far as the few rows of `r.seqs` sequences leave
    // SMs idle, of two CTAs where a launch may hold many rows
    const long U = (long)p.G * r.seqs * attn_units(std::min(r.most, (r.total + r.seqs - 1) / r.seqs), rep, 8);
    while (a.S < 8 && 2 * a.S <= nb && U * 2 * a.S <= p.sms) a.S *= 2;
    if (a.S == 1 && nb >= 4) a.S = 2;
    a.mode = ATTN_BY_ROWS;
    a.clusters = (long)p.G * (attn_units(r.total, rep, 4) + p.batch);
  }
  a.clusters = std::min<long>(a.clusters, std::max(1, p.sms / a.S));
  return a;
}

template <int HD>
cudaError_t launch_attn(const AttnPlan& p, const AttnRows& rows, int* err, cudaStream_t stream) {
  static bool attr_set = false;
  auto kern = attn_tc_kernel<HD>;
  if (!attr_set) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AttnCfg<HD>::SMEM);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  const AttnShape a = attn_shape(p, rows);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.S * a.clusters));
  cfg.blockDim = dim3(AT_THREADS);
  cfg.dynamicSmemBytes = AttnCfg<HD>::SMEM;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = a.S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, p.tq, p.tk, p.tv, p.to, p.out, p.batch, p.T, p.H, p.G, p.H / p.G, p.kcol0, p.seq_off,
                            p.seq_len, rows.most, a.mode, a.bands, 1.0f / (float)p.sms, err);
}

}  // namespace

int attn_vt_pitch(int T) { return (T + 7) & ~7; }

cudaError_t attention_plan(AttnPlan* p, const __nv_bfloat16* qkv, const __nv_bfloat16* kbuf, __half* vt,
                           __nv_bfloat16* out, int batch, int T, int H, int G, int hd, int rows_max,
                           const int* seq_off, const int* seq_len, int num_sms) {
  if (num_sms <= 0 || batch <= 0 || T <= 0 || H <= 0 || G <= 0 || H % G || (hd != 64 && hd != 128) || rows_max <= 0)
    return cudaErrorInvalidValue;
  if ((reinterpret_cast<uintptr_t>(qkv) & 15) || (reinterpret_cast<uintptr_t>(vt) & 15) ||
      (reinterpret_cast<uintptr_t>(out) & 15) || (kbuf && (reinterpret_cast<uintptr_t>(kbuf) & 15)))
    return cudaErrorInvalidValue;
  const uint64_t cols = (uint64_t)(H + 2 * G) * hd, ocols = (uint64_t)H * hd, Tp = attn_vt_pitch(T);
  {  // q rows of the step, a band at a time: [rows_max][cols]
    const uint64_t dims[2] = {cols, (uint64_t)rows_max};
    const uint64_t strides[1] = {cols * 2};
    const uint32_t box[2] = {64, 32};
    if (!encode_tmap(&p->tq, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(qkv), dims, strides, box,
                     CU_TENSOR_MAP_SWIZZLE_128B))
      return cudaErrorInvalidValue;
  }
  {  // keys of every position as [batch][T][kcols]: the key store, or the k columns of q|k|v
    const uint64_t kcols = kbuf ? (uint64_t)G * hd : cols;
    const uint64_t dims[3] = {kcols, (uint64_t)T, (uint64_t)batch};
    const uint64_t strides[2] = {kcols * 2, (uint64_t)T * kcols * 2};
    const uint32_t box[3] = {64, 128, 1};
    if (!encode_tmap(&p->tk, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16*>(kbuf ? kbuf : qkv), dims,
                     strides, box, CU_TENSOR_MAP_SWIZZLE_128B))
      return cudaErrorInvalidValue;
    p->kcol0 = kbuf ? 0 : H * hd;
  }
  {  // v^T as [batch*G][hd][T] (row pitch Tp)
    const uint64_t dims[3] = {(uint64_t)T, (uint64_t)hd, (uint64_t)batch * G};
    const uint64_t strides[2] = {Tp * 2, (uint64_t)hd * Tp * 2};
    const uint32_t box[3] = {64, (uint32_t)hd, 1};
    if (!encode_tmap(&p->tv, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, vt, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B))
      return cudaErrorInvalidValue;
  }
  if (seq_off) {  // output rows of the step: [rows_max][H*hd] (32-row bands of one sequence)
    const uint64_t dims[2] = {ocols, (uint64_t)rows_max};
    const uint64_t strides[1] = {ocols * 2};
    const uint32_t box[2] = {64, 32};
    if (!encode_tmap(&p->to, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, out, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B))
      return cudaErrorInvalidValue;
  } else {  // [batch][T][H*hd]: stores of rows past T are clipped
    const uint64_t dims[3] = {ocols, (uint64_t)T, (uint64_t)batch};
    const uint64_t strides[2] = {ocols * 2, (uint64_t)T * ocols * 2};
    const uint32_t box[3] = {64, 32, 1};
    if (!encode_tmap(&p->to, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, out, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B))
      return cudaErrorInvalidValue;
  }
  p->qkv = qkv;
  p->out = out;
  p->vt = vt;
  p->seq_off = seq_off;
  p->seq_len = seq_len;
  p->batch = batch;
  p->T = T;
  p->H = H;
  p->G = G;
  p->hd = hd;
  p->sms = num_sms;
  return cudaSuccess;
}

cudaError_t attention_transpose_launch(const AttnPlan& p, cudaStream_t stream) {
  const int cols = (p.H + 2 * p.G) * p.hd, ghd = p.G * p.hd;
  dim3 tgrid((attn_vt_pitch(p.T) + 63) / 64, (ghd + 63) / 64, p.batch);
  return launch_pdl(v_transpose_kernel, tgrid, 256, 0, stream, p.qkv, p.vt, p.T, attn_vt_pitch(p.T), cols,
                    (p.H + p.G) * p.hd, ghd);
}

cudaError_t attention_core_launch(const AttnPlan& p, const AttnRows& rows, int* err, cudaStream_t stream) {
  return p.hd == 128 ? launch_attn<128>(p, rows, err, stream) : launch_attn<64>(p, rows, err, stream);
}

cudaError_t attention_launch(const AttnPlan& p, const AttnRows& rows, int* err, cudaStream_t stream) {
  const cudaError_t e = attention_transpose_launch(p, stream);
  return e != cudaSuccess ? e : attention_core_launch(p, rows, err, stream);
}

}  // namespace dcl
