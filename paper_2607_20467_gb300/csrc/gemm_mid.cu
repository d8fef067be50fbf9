// GEMMs of a step with a middling number of rows (more than the few-row kernel takes):
//   out = X[rows][K] @ W[N][K]^T   with the layer epilogues fused,
// as the CTA-pair kernel of gemm_tc.cu but with the operands swapped: 256 weight rows on the
// MMA's M side (128 per CTA of the pair) and a tile of nt tokens on its N side.
//
// With the tokens on the M side every 256-row block costs a whole one: 544 rows (a suffix of
// the long generation under the prefix cache) pay for 768.  On the N side a tile is any multiple
// of 32 up to 256 tokens, so the MMA time follows the rows, and the tile is also what balances
// the rounds: the tokens are cut into `tt` tiles and K into `splits` ranges (residual epilogue
// only, added in order) such that rounds of items x item length is least (mid_shape, one entry
// per 32 rows, computed by the host).
//
// One persistent CTA pair per two SMs, 192 threads per CTA: TMA producer (both CTAs), MMA issuer
// (the leader's warp 1), four epilogue warps.  The accumulator is double-buffered in TMEM; the
// epilogue brings 32 tokens at a time through shared memory (a lane holds a weight row, an
// output row is a token) while the next item's products run.
#include <string.h>

#include <algorithm>

#include "common.cuh"
#include "few_epi.cuh"
#include "tc_ptx.cuh"

namespace dcl {
namespace {

constexpr int MD_THREADS = 192;
constexpr int MD_BK = 64;
constexpr int MD_W_BYTES = 128 * 128;      // a CTA's 128 weight rows of one K block
constexpr int MD_STAGE_BYTES = 2 * MD_W_BYTES;  // and up to 128 tokens
constexpr int MD_STAGES = 6;
constexpr int MD_MORE_TILES = 2;           // tiles of tokens beyond the fewest
constexpr int MD_CHUNK = 32;               // tokens staged at a time
constexpr int MD_STG = MD_CHUNK * FW_PITCH * 4;
constexpr int MD_BARS = 256 + 2 * 4 * MD_CHUNK;
constexpr size_t MD_SMEM = 1024 + (size_t)MD_STAGES * MD_STAGE_BYTES + MD_STG + MD_BARS;
static_assert(MD_SMEM <= 232448, "shared memory per CTA");
static_assert(8 * (2 * MD_STAGES + 5) + 8 <= 256, "barrier area");

struct MidArgs {
  FewArgs f;
  const uint16_t* shapes;  // by rows / 32 rounded up: tt + 256 * splits
  int pair_units;          // tiles of 256 weight rows
  int* flags;              // [tiles][2] ordered-add counters, zero between launches (splits > 1)
};

struct MidItem {
  int u2, tk, sp, kb0, kb1;
};

template <int EPI>
__global__ void __launch_bounds__(MD_THREADS, 1)
    mid_gemm_kernel(const __grid_constant__ CUtensorMap tw, const __grid_constant__ MidTokens tx,
                    const __grid_constant__ MidArgs a, int* err) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  const uint32_t stg = base + MD_STAGES * MD_STAGE_BYTES;
  const uint32_t bars = stg + MD_STG;
  const uint32_t full0 = bars, empty0 = bars + 8 * MD_STAGES, tfull0 = empty0 + 8 * MD_STAGES, tempty0 = tfull0 + 16;
  const uint32_t drain = tempty0 + 16, holder = drain + 8;
  volatile uint32_t* holder_ptr = reinterpret_cast<volatile uint32_t*>(smem + (holder - base));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + (holder + 4 - base));
  int* pos_s = reinterpret_cast<int*>(smem + (bars + 256 - base));
  int* seq_s = pos_s + MD_CHUNK;

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank();  // 0: the pair's leader
  const int c = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < MD_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(tfull0 + 8 * i, 1);
      mbar_init(tempty0 + 8 * i, 8);  // 4 epilogue warps x 2 CTAs (used in the leader)
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tw);
    for (int i = 0; i < 8; ++i) prefetch_tmap(&tx.box[i]);
  }
  if (warp == 1) tmem_alloc_pair(holder, 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the peer's barriers exist before any remote arrive
  tc_fence_after();
  const uint32_t tmem_base = *holder_ptr;
  pdl_wait();
  pdl_launch_dependents();

  const int rows = a.f.ep.m_dev ? min(a.f.M, *a.f.ep.m_dev) : a.f.M;
  const int shape = a.shapes[(rows + 31) >> 5];
  const int tt = shape & 255, S = shape >> 8;
  const int per = tt ? (rows + tt - 1) / tt : 0, nt = min((per + 31) & ~31, 256);  // tokens of a tile
  const int tiles = a.pair_units * tt, items = nt * tt >= rows ? tiles * S : 0;
  if (rows > 0 && items == 0 && threadIdx.x == 0) report_error(err, DERR_BAD_SHAPE);
  auto item = [&](int idx, MidItem& it) -> bool {
    const int w = c + idx * pairs;
    if (w >= items) return false;
    it.sp = w / tiles;
    const int r = w - it.sp * tiles;
    it.u2 = r / tt;
    it.tk = r - it.u2 * tt;
    it.kb0 = it.sp * a.f.nkb / S;
    it.kb1 = (it.sp + 1) * a.f.nkb / S;
    return true;
  };
  // an item's tokens on the MMA's N side (the last tile of tokens may be shorter)
  auto width = [&](const MidItem& it) { return min(nt, (max(rows - it.tk * nt, 1) + 31) & ~31); };

  if (warp == 0) {
    // ------------------------------------------------ TMA producer (both CTAs; the whole warp,
    // one lane issues: a diverged thread took 86 cycles a box)
    const bool leader = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    MidItem it;
    for (int idx = 0; ok && item(idx, it); ++idx) {
      const int half = width(it) / 2, x0 = it.tk * nt + rank * half;
      const CUtensorMap* tokens = &tx.box[half / 16 - 1];
      for (int kb = it.kb0; kb < it.kb1; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait_inline(empty0 + 8 * stage, phase ^ 1u, abort_flag))) {
          ok = false;
          break;
        }
        if (leader) {
          const uint32_t full_leader = map_cluster(full0 + 8 * stage, 0);
          if (rank == 0) mbar_arrive_expect_tx(full0 + 8 * stage, 2u * (uint32_t)(MD_W_BYTES + half * 128));
          const uint32_t dst = base + (uint32_t)(stage * MD_STAGE_BYTES);
          if constexpr (EPI == EPI_SWIGLU) {  // 64 gate rows and the matching 64 up rows (128 rows apart)
            tma_load_2d_pair(dst, &tw, kb * MD_BK, it.u2 * 256 + rank * 64, full_leader);
            tma_load_2d_pair(dst + MD_W_BYTES / 2, &tw, kb * MD_BK, it.u2 * 256 + 128 + rank * 64, full_leader);
          } else {
            tma_load_2d_pair(dst, &tw, kb * MD_BK, it.u2 * 256 + rank * 128, full_leader);
          }
          tma_load_2d_pair(dst + MD_W_BYTES, tokens, kb * MD_BK, x0, full_leader);
        }
        __syncwarp();
        if (++stage == MD_STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok) {
      *abort_flag = 1;
      if (leader) report_error(err, DERR_WAIT_TIMEOUT);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ------------------------------------------------ MMA issuer (the whole warp, one lane issues)
      const bool leader = elect_one();
      auto wait = [&](uint32_t bar, uint32_t parity) {
        return (bool)__all_sync(0xffffffffu, mbar_wait_inline(bar, parity, abort_flag));
      };
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      MidItem it;
      for (int idx = 0; ok && item(idx, it); ++idx) {
        const int ab = idx & 1;
        const uint32_t idesc = make_idesc(256, width(it));
        if (!wait(tempty0 + 8 * ab, ((uint32_t)(idx >> 1) & 1u) ^ 1u)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(ab * 256);
        for (int kb = it.kb0; kb < it.kb1; ++kb) {
          if (!wait(full0 + 8 * stage, phase)) {
            ok = false;
            break;
          }
          if (leader) {
            const uint32_t sw = base + (uint32_t)(stage * MD_STAGE_BYTES);
            const uint64_t dw = sw128_desc(sw), dx = sw128_desc(sw + MD_W_BYTES);
#pragma unroll
            for (int k = 0; k < MD_BK / 16; ++k)
              umma_bf16_pair(d_tmem, dw + 2 * k, dx + 2 * k, idesc, (kb > it.kb0 || k > 0) ? 1u : 0u);
            umma_commit_pair(empty0 + 8 * stage, 3);
          }
          __syncwarp();
          if (++stage == MD_STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        if (leader) umma_commit_pair(tfull0 + 8 * ab, 3);
        __syncwarp();
      }
      if (!ok) {
        *abort_flag = 1;
        if (leader) report_error(err, DERR_WAIT_TIMEOUT);
      }
      if (leader) umma_commit_pair(drain, 1);
      __syncwarp();
      volatile int no_abort = 0;
      mbar_wait(drain, 0, &no_abort);
    }
  } else {
    // ------------------------------------------------ epilogue warps 2..5 (both CTAs)
    const int q = warp & 3;  // TMEM lane quarter: weight rows 32 q .. 32 q + 31 of this CTA's 128
    const int et = (int)threadIdx.x - 64;
    bool ok = true;  // (after a failed wait a warp still meets the others at every barrier of its items)
    MidItem it;
    for (int idx = 0; item(idx, it); ++idx) {
      const int ab = idx & 1;
      if (ok && !__all_sync(0xffffffffu, mbar_wait(tfull0 + 8 * ab, (uint32_t)(idx >> 1) & 1u, abort_flag))) {
        ok = false;
        *abort_flag = 1;
        report_error(err, DERR_WAIT_TIMEOUT);
      }
      tc_fence_after();
      const int tok0 = it.tk * nt, n = min(nt, rows - tok0), u = 2 * it.u2 + rank;
      int* flag = a.flags + (it.u2 * tt + it.tk) * 2 + rank;
      if (S > 1) {  // split sp is added to the residual stream after split sp - 1
        if (et == 0 && !wait_flag_geq(flag, it.sp, abort_flag)) {
          *abort_flag = 1;
          report_error(err, DERR_WAIT_TIMEOUT);
        }
        epilogue_bar();
      }
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * 256);
#pragma unroll 1
      for (int t0 = 0; t0 < n; t0 += MD_CHUNK) {
        if (EPI == EPI_QKV_ROPE && et < MD_CHUNK && t0 + et < n) {
          pos_s[et] = a.f.ep.row_pos[tok0 + t0 + et];
          seq_s[et] = a.f.ep.row_seq[tok0 + t0 + et];
        }
        if (ok) {
          uint32_t v[32];
          tmem_ld32(taddr + (uint32_t)t0, v);
          tmem_ld_wait();
          const uint32_t at = stg + (uint32_t)(q * 32 + lane) * 4;
#pragma unroll
          for (int i = 0; i < 32; ++i) st_shared_f32(at + (uint32_t)(i * FW_PITCH * 4), f32(v[i]));
        }
        if (t0 + MD_CHUNK >= n) {  // the accumulator has been read
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(map_cluster(tempty0 + 8 * ab, 0));
        }
        epilogue_bar();
        if (!*abort_flag) few_finish<EPI, 1>(a.f, stg, u, tok0 + t0, 0, min(MD_CHUNK, n - t0), et, pos_s, seq_s);
        epilogue_bar();  // the staged sums have been read
      }
      if (n <= 0) {  // (a tile past the rows: its accumulator is free too)
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_cluster(tempty0 + 8 * ab, 0));
      }
      if (S > 1) {
        __threadfence();
        epilogue_bar();
        if (et == 0) atomicExch(flag, it.sp + 1 == S ? 0 : it.sp + 1);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (*abort_flag) abort_grace();
  __syncwarp();
  cluster_sync();  // no CTA leaves while its pair may still touch its smem or TMEM
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

template <int EPI>
cudaError_t launch_mid(const MidPlan& p, int* err, cudaStream_t stream) {
  static bool attr_set = false;
  auto kern = mid_gemm_kernel<EPI>;
  if (!attr_set) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MD_SMEM);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  MidArgs a;
  a.f.nkb = p.K / MD_BK;
  a.f.N = p.N;
  a.f.M = p.M;
  a.f.ep = p.ep;
  a.shapes = p.shapes;
  a.pair_units = p.N / 256;
  a.flags = p.flags;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.grid);
  cfg.blockDim = dim3(MD_THREADS);
  cfg.dynamicSmemBytes = MD_SMEM;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, p.tw, p.tx, a, err);
}

}  // namespace

// Fitted to 160 .. 1536 rows of the LLaDA-8B and Dream-7B shapes with tiles of 64 .. 256 tokens:
// a K block of nt tokens against one of 256 (the loads of the weights do not shrink with nt), a
// launch's start and end, and for each part of a split the wait for the one before.
MidShape mid_shape(int rows, int N, int K, int epi, int pairs) {
  MidShape best;
  const int units = N / 256, nkb = K / MD_BK, t0 = (rows + 255) / 256;
  for (int tt = t0; tt <= t0 + MD_MORE_TILES && tt <= 255; ++tt) {
    const int nt = std::min(((rows + tt - 1) / tt + 31) / 32 * 32, 256);
    if (tt > 1 && nt * (tt - 1) >= rows) continue;  // (a tile would be empty)
    for (int S = 1; S <= (epi == EPI_RESID_F32 ? 6 : 1) && S <= nkb; ++S) {
      const long rounds = ((long)units * tt * S + pairs - 1) / pairs;
      const double x = nt / 256.0, block = std::max(0.25 + 0.75 * x, 0.45 + 0.45 * x);
      const double cost = (double)rounds * ((nkb + S - 1) / S) * block + 15.0 + (S > 1 ? 6.0 * S : 0.0);
      if (best.tt == 0 || cost < best.cost) best = {tt, S, cost};
    }
  }
  return best;
}

cudaError_t mid_plan(MidPlan* p, const void* X, int M, int K, const void* W, int N, int epi, const FewEpi& ep,
                     int num_sms) {
  if (M <= 0 || N <= 0 || K <= 0 || K % MD_BK || N % 256 || num_sms < 2 || M > 255 * 256) return cudaErrorInvalidValue;
  if ((reinterpret_cast<uintptr_t>(X) & 15) || (reinterpret_cast<uintptr_t>(W) & 15) ||
      (reinterpret_cast<uintptr_t>(ep.out) & 15) || ep.ldo % 4)
    return cudaErrorInvalidValue;
  if (epi != EPI_RESID_F32 && epi != EPI_QKV_ROPE && epi != EPI_SWIGLU) return cudaErrorInvalidValue;
  if (epi == EPI_QKV_ROPE && ((ep.head_dim != 64 && ep.head_dim != 128) || ep.rope_cols % FW_TILE || N % ep.head_dim ||
                              (ep.kdst && ep.k_col0 % FW_TILE)))
    return cudaErrorInvalidValue;
  const uint64_t wd[2] = {(uint64_t)K, (uint64_t)N}, xd[2] = {(uint64_t)K, (uint64_t)M}, st[1] = {(uint64_t)K * 2};
  const uint32_t wb[2] = {MD_BK, epi == EPI_SWIGLU ? 64u : 128u};
  if (!encode_tmap(&p->tw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(W), wd, st, wb,
                   CU_TENSOR_MAP_SWIZZLE_128B))
    return cudaErrorInvalidValue;
  for (int i = 0; i < 8; ++i) {
    const uint32_t xb[2] = {MD_BK, 16u * (i + 1)};
    if (!encode_tmap(&p->tx.box[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(X), xd, st, xb,
                     CU_TENSOR_MAP_SWIZZLE_128B))
      return cudaErrorInvalidValue;
  }
  p->M = M;
  p->N = N;
  p->K = K;
  p->epi = epi;
  p->ep = ep;
  p->grid = num_sms / 2 * 2;
  p->flags_needed = (size_t)(N / 256) * ((M + 255) / 256 + MD_MORE_TILES) * 2;
  return cudaSuccess;
}

cudaError_t mid_launch(const MidPlan& p, int* err, cudaStream_t stream) {
  if (!p.flags || !p.shapes) return cudaErrorInvalidValue;
  switch (p.epi) {
    case EPI_RESID_F32: return launch_mid<EPI_RESID_F32>(p, err, stream);
    case EPI_QKV_ROPE: return launch_mid<EPI_QKV_ROPE>(p, err, stream);
    case EPI_SWIGLU: return launch_mid<EPI_SWIGLU>(p, err, stream);
  }
  return cudaErrorInvalidValue;
}

}  // namespace dcl
