// GEMMs of a step with few rows (the current block or a short
// suffix under the key / value caches, small full recomputes):
//   out = X[rows][K] @ W[N][K]^T   with the step's epilogues fused.
//
// What bounds them is the weight stream: every weight is read once for a handful of tokens.
// The CTA-pair kernel puts tokens on the MMA's 256-row side, so that 32 live rows cost the
// MMA time of 256 (18 us per 256 x 256 x 4096 tile) on as many SM pairs as there are column
// tiles (48 of 76 for QKV, 16 for O).  Here the operands are swapped: 128 weight rows on the
// M side, the tokens (rounded up to 32) on the N side, so the MMA time follows the tokens, and
// each tile of 128 weight rows is split by K over a cluster of S CTAs, as far as the grid stays
// within two CTAs per SM and the shares are worth it (few_plan).
//
// One CTA = one tile's share of K (192 threads: TMA producer, MMA issuer, four epilogue
// warps).  Its fp32 sum goes from TMEM to its idle operand ring; after a cluster barrier each
// CTA of the cluster finishes nt / S tokens, adding the S sums through distributed shared
// memory in K order (bit-reproducible), so the tail is a barrier and one short pass (about 2.5
// us) instead of a round trip of partial sums through L2 (which made these launches no faster
// than the pair kernel's).
//
// A CTA takes less than half of an SM's shared memory, TMEM and registers, so that under
// programmatic dependent launch the next GEMM of the step is resident beside the running one
// and fills its ring with weights, which depend on no earlier kernel, before its
// dependent-launch wait: the HBM keeps streaming across kernel boundaries.  More CTAs (more
// bytes in flight) stream faster: 192 CTAs of the gate/up GEMM read 201 MB in 29 us (6.9
// TB/s), 96 CTAs of an unsplit QKV 100 MB in 22 us, 192 in 16 us.
//
// Where the weights are small (few_rows) more rows are taken too, as tiles of 128 tokens beside
// each other: while all tiles fit the GPU at once a launch is latency, and these are shorter
// than the pair kernel's (a fused MLP took 27 us at d 768, ffn 2048).
//
// Measured per step, 8 layers of the LLaDA-8B shape at T = 1536: 32 rows 1415 -> 1092 us, 96
// rows 1430 -> 1208 us; the 2-layer test model (96 rows, latency) 119 -> 81 us; four layers of
// d 768, ffn 2048: 192 rows 254 -> 214 us, 512 rows 260 -> 231, 1024 rows 278 -> 243 (at 1536
// rows, past one round of tiles, the pair kernels take 299).
#include <string.h>

#include <algorithm>

#include "common.cuh"
#include "few_epi.cuh"
#include "tc_ptx.cuh"

namespace dcl {
namespace {

constexpr int FW_THREADS = 192;
constexpr int FW_BK = 64;                 // K block: one 128-byte swizzle row of bf16
constexpr int FW_W_BYTES = FW_TILE * 128; // a K block of them
constexpr int FW_XBOX_BYTES = 32 * 128;   // 32 tokens x one K block
constexpr int FW_MAX_STAGES = 5;
constexpr int FW_BARS = 256 + 2 * 4 * FEW_TILE_ROWS;  // barriers, then the tokens' positions and sequences
constexpr size_t FW_SMEM = 112 * 1024;
constexpr int FW_RING = (int)FW_SMEM - 1024 - FW_BARS;
static_assert(FEW_TILE_ROWS * FW_PITCH * 4 <= FW_RING, "the staged sum lives in the operand ring");
static_assert(8 * (2 * FW_MAX_STAGES + 1) + 16 <= 256, "barrier area");

struct FewTiles {
  int nt_max;        // tokens of a token tile at most (32 or FEW_TILE_ROWS)
  int units, tiles;  // tiles of weight rows, of tokens
};

template <int EPI>
__global__ void __launch_bounds__(FW_THREADS, 2)
    few_gemm_kernel(const __grid_constant__ CUtensorMap tw, const __grid_constant__ CUtensorMap tx,
                    const __grid_constant__ FewArgs a, const FewTiles cut, int* err) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  const uint32_t bars = base + FW_RING;
  const uint32_t full0 = bars, empty0 = bars + 8 * FW_MAX_STAGES, done = empty0 + 8 * FW_MAX_STAGES, holder = done + 8;
  volatile uint32_t* holder_ptr = reinterpret_cast<volatile uint32_t*>(smem + (holder - base));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + (holder + 4 - base));
  int* pos_s = reinterpret_cast<int*>(smem + FW_RING + 256);
  int* seq_s = pos_s + FEW_TILE_ROWS;

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // (warp-uniform)
  const int S = (int)cluster_size(), rank = (int)cluster_rank();
  // the cluster's tile of weight rows and its tile of tokens (rows [tok0, tok0 + nt_max))
  const int u = (int)blockIdx.x / S % cut.units, tok0 = (int)blockIdx.x / S / cut.units * cut.nt_max;
  const int kb0 = rank * a.nkb / S, nkb = (rank + 1) * a.nkb / S - kb0;
  // a stage: the weight rows of one K block, then the tokens'.  The stage pitch is that of
  // the most tokens the launch may hold, known before the row count is.
  const int stage_bytes = FW_W_BYTES + cut.nt_max * 128;
  const int stages = min(FW_RING / stage_bytes, FW_MAX_STAGES);

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tw);
    prefetch_tmap(&tx);
  }

  auto load_w = [&](int stage, int kb) {
    const uint32_t dst = base + (uint32_t)(stage * stage_bytes), bar = full0 + 8 * stage;
    if constexpr (EPI == EPI_SWIGLU) {  // 64 gate rows and the matching 64 up rows (128 rows apart)
      const int row = (u >> 1) * 256 + (u & 1) * 64;
      tma_load_2d(dst, &tw, (kb0 + kb) * FW_BK, row, bar);
      tma_load_2d(dst + FW_W_BYTES / 2, &tw, (kb0 + kb) * FW_BK, row + 128, bar);
    } else {
      tma_load_2d(dst, &tw, (kb0 + kb) * FW_BK, u * FW_TILE, bar);
    }
  };
  // the first stages' weights, before the dependent-launch wait (no kernel of the step writes them)
  const int pre = a.ep.w_early ? min(stages, nkb) : 0;
  if (threadIdx.x == 0)
    for (int kb = 0; kb < pre; ++kb) {
      mbar_expect_tx(full0 + 8 * kb, FW_W_BYTES);
      load_w(kb, kb);
    }
  if (warp == 1) tmem_alloc(holder, FEW_TILE_ROWS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *holder_ptr;

  pdl_wait();
  pdl_launch_dependents();
  const int all = a.ep.m_dev ? min(a.M, *a.ep.m_dev) : a.M;
  const int rows = max(min(all - tok0, cut.nt_max), 0);
  int nt = (rows + 31) & ~31;         // the MMA's N
  if (all > cut.tiles * cut.nt_max) {     // (the launch is not chosen for so many rows)
    if (threadIdx.x == 0) report_error(err, DERR_BAD_SHAPE);
    nt = 0;
  }

  if (warp == 0) {
    // ------------------------------------------------ TMA producer (the whole warp, one lane issues)
    const bool leader = elect_one();
    bool ok = true;
    int issued = 0, stage = 0;
    uint32_t phase = 0;
    for (int kb = 0; kb < (nt > 0 ? nkb : pre); ++kb) {
      const bool have_w = kb < pre;
      if (!have_w && !__all_sync(0xffffffffu, mbar_wait_inline(empty0 + 8 * stage, phase ^ 1u, abort_flag))) {
        ok = false;
        break;
      }
      if (leader) {
        mbar_arrive_expect_tx(full0 + 8 * stage, (have_w ? 0 : FW_W_BYTES) + nt * 128);
        if (!have_w) load_w(stage, kb);
        for (int b = 0; b < nt / 32; ++b)
          tma_load_2d(base + (uint32_t)(stage * stage_bytes + FW_W_BYTES + b * FW_XBOX_BYTES), &tx, (kb0 + kb) * FW_BK,
                      tok0 + b * 32, full0 + 8 * stage);
      }
      __syncwarp();
      ++issued;
      if (++stage == stages) {
        stage = 0;
        phase ^= 1u;
      }
    }
    if (!ok) {
      *abort_flag = 1;
      if (leader) report_error(err, DERR_WAIT_TIMEOUT);
    }
    if (!ok || nt == 0) {  // every copy issued lands before the CTA leaves (bounded)
      for (int s = 0; s < stages && s < issued; ++s) {
        const int arms = (issued - 1 - s) / stages + 1;
        volatile int no_abort = 0;
        mbar_wait(full0 + 8 * s, (uint32_t)((arms - 1) & 1), &no_abort);
      }
    }
  } else if (warp == 1) {
    if (nt > 0) {
      // ------------------------------------------------ MMA issuer (the whole warp, one lane issues)
      const uint32_t idesc = make_idesc(FW_TILE, nt);
      const bool leader = elect_one();
      bool ok = true;
      int stage = 0;
      uint32_t phase = 0;
      for (int kb = 0; kb < nkb; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait_inline(full0 + 8 * stage, phase, abort_flag))) {
          ok = false;
          break;
        }
        if (leader) {
          const uint32_t sw = base + (uint32_t)(stage * stage_bytes);
          const uint64_t dw = sw128_desc(sw), dx = sw128_desc(sw + FW_W_BYTES);
#pragma unroll
          for (int k = 0; k < FW_BK / 16; ++k)
            umma_bf16(tmem_base, dw + 2 * k, dx + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          umma_commit(empty0 + 8 * stage);
        }
        __syncwarp();
        if (++stage == stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!ok) {
        *abort_flag = 1;
        if (leader) report_error(err, DERR_WAIT_TIMEOUT);
      }
      if (leader) umma_commit(done);  // (in either case every MMA issued here completes before TMEM is released)
      __syncwarp();
      volatile int no_abort = 0;
      mbar_wait(done, 0, &no_abort);
    }
  } else if (nt > 0) {
    // ------------------------------------------------ epilogue warps 2..5: the sum to shared memory
    const int et = threadIdx.x - 64;
    if (EPI == EPI_QKV_ROPE && et < rows) {
      pos_s[et] = a.ep.row_pos[tok0 + et];
      seq_s[et] = a.ep.row_seq[tok0 + et];
    }
    const int q = warp & 3;  // TMEM lane quarter: rows 32 q .. 32 q + 31 of the tile
    bool ok = mbar_wait(done, 0, abort_flag);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) {
      *abort_flag = 1;
      report_error(err, DERR_WAIT_TIMEOUT);
    } else {
      tc_fence_after();
#pragma unroll 1
      for (int t0 = 0; t0 < nt; t0 += 32) {
        uint32_t v[32];
        tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)t0, v);
        tmem_ld_wait();
        const uint32_t at = base + (uint32_t)(t0 * FW_PITCH + q * 32 + lane) * 4;
#pragma unroll
        for (int i = 0; i < 32; ++i) st_shared_f32(at + (uint32_t)(i * FW_PITCH * 4), f32(v[i]));
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, FEW_TILE_ROWS);
  }
  if (S > 1) cluster_sync();  // every CTA of the cluster has its sum in shared memory
  if (warp >= 2 && nt > 0 && !*abort_flag) {
    const int t0 = rank * nt / S, t1 = min((rank + 1) * nt / S, rows);
    const int et = threadIdx.x - 64;
    switch (S) {
      case 1: few_finish<EPI, 1>(a, base, u, tok0, t0, t1, et, pos_s, seq_s); break;
      case 2: few_finish<EPI, 2>(a, base, u, tok0, t0, t1, et, pos_s, seq_s); break;
      case 4: few_finish<EPI, 4>(a, base, u, tok0, t0, t1, et, pos_s, seq_s); break;
      case 8: few_finish<EPI, 8>(a, base, u, tok0, t0, t1, et, pos_s, seq_s); break;
    }
  }
  __syncwarp();
  if (S > 1) cluster_sync_relaxed();  // no CTA leaves while another may read its sum
}

bool encode_2d(CUtensorMap* tm, const void* p, int rows, int k, int box_rows) {
  const uint64_t dims[2] = {(uint64_t)k, (uint64_t)rows};
  const uint64_t strides[1] = {(uint64_t)k * 2};
  const uint32_t box[2] = {FW_BK, (uint32_t)box_rows};
  return encode_tmap(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(p), dims, strides, box,
                     CU_TENSOR_MAP_SWIZZLE_128B);
}

template <int EPI>
cudaError_t launch_few(const FewPlan& p, int* err, cudaStream_t stream) {
  static bool attr_set = false;
  auto kern = few_gemm_kernel<EPI>;
  if (!attr_set) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FW_SMEM);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  FewArgs a;
  a.nkb = p.K / FW_BK;
  a.N = p.N;
  a.M = p.M;
  a.ep = p.ep;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.units * p.tiles * p.split);
  cfg.blockDim = dim3(FW_THREADS);
  cfg.dynamicSmemBytes = FW_SMEM;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.split;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, p.tw, p.tx, a, FewTiles{p.nt_max, p.units, p.tiles}, err);
}

}  // namespace

cudaError_t few_plan(FewPlan* p, const void* X, int M, int K, const void* W, int N, int epi, const FewEpi& ep,
                     int num_sms, int rows) {
  const int nt_max = rows <= 32 ? 32 : FEW_TILE_ROWS;
  if (M <= 0 || N <= 0 || K <= 0 || K % FW_BK || rows <= 0) return cudaErrorInvalidValue;
  if ((reinterpret_cast<uintptr_t>(X) & 15) || (reinterpret_cast<uintptr_t>(W) & 15) ||
      (reinterpret_cast<uintptr_t>(ep.out) & 15) || ep.ldo % 4 || N % 4)
    return cudaErrorInvalidValue;
  switch (epi) {
    case EPI_BF16:
    case EPI_RESID_F32: break;
    case EPI_SWIGLU:
      if (N % 256) return cudaErrorInvalidValue;
      break;
    case EPI_QKV_ROPE:  // whole heads in a tile, each tile all q, all k or all v
      if ((ep.head_dim != 64 && ep.head_dim != 128) || ep.rope_cols % FW_TILE || N % ep.head_dim ||
          (ep.kdst && ep.k_col0 % FW_TILE))
        return cudaErrorInvalidValue;
      break;
    default: return cudaErrorInvalidValue;
  }
  if (!encode_2d(&p->tw, W, N, K, epi == EPI_SWIGLU ? FW_TILE / 2 : FW_TILE) || !encode_2d(&p->tx, X, M, K, 32))
    return cudaErrorInvalidValue;
  p->M = M;
  p->N = N;
  p->K = K;
  p->epi = epi;
  p->ep = ep;
  p->nt_max = nt_max;
  p->units = (N + FW_TILE - 1) / FW_TILE;
  p->tiles = (rows + nt_max - 1) / nt_max;
  // (at least this many K blocks for each CTA of a split: the cluster's barrier and its reads of
  // distributed shared memory cost more than a shorter share saves.  d 768, ffn 2048, 384 rows,
  // four layers: 222 us a step with splits down to one block, 206 with two and 196 so; a long K
  // is a weight stream, which wants all eight)
  const int nkb = K / FW_BK;
  auto fits = [&](int S) {
    return p->units * p->tiles * S <= 2 * num_sms && nkb / S >= (S == 2 ? 2 : S == 4 ? 3 : 8);
  };
  p->split = 1;
  while (p->split < 8 && fits(2 * p->split)) p->split *= 2;
  return cudaSuccess;
}

int few_rows(int N, int num_sms) {
  return FEW_TILE_ROWS * std::max(1, 2 * num_sms / ((N + FW_TILE - 1) / FW_TILE));
}

cudaError_t few_launch(const FewPlan& p, int* err, cudaStream_t stream) {
  switch (p.epi) {
    case EPI_BF16: return launch_few<EPI_BF16>(p, err, stream);
    case EPI_RESID_F32: return launch_few<EPI_RESID_F32>(p, err, stream);
    case EPI_QKV_ROPE: return launch_few<EPI_QKV_ROPE>(p, err, stream);
    case EPI_SWIGLU: return launch_few<EPI_SWIGLU>(p, err, stream);
  }
  return cudaErrorInvalidValue;
}

}  // namespace dcl
