// lmhead.cu -- the target's greedy prediction per node straight from its final
// hidden states: logits = H W^T (the LM head), reduced to their argmax inside
// the GEMM's epilogue, so the logits never reach HBM (paper Sec. 2
// "Speculative decoding" at temperature 0; the logits are the target's
// per-node distribution that the acceptance reads).
//
// tcgen05 GEMM, persistent, on pairs of CTAs (cta_group::2, two SMs). A tile is
// 256 vocabulary entries (the MMA's M side, 128 per CTA) by up to 256 rows of H
// (its N side, of which each CTA loads half), so that a 64-column block of the
// largest tile costs each SM 32 KB from L2 for its 128 x 256 share, where a CTA
// by itself reads 48 KB, and few rows cost no padding to 128. 320 threads per CTA:
//   warp 0, one thread  TMA producer: this CTA's halves of W and H, two blocks
//                       of 64 columns (128-byte swizzle) per ring stage
//   warp 1, converged   in the even CTA the MMA issuer (M256 K16, bf16 -> f32)
//                       into one of two TMEM accumulators of 256 columns; its
//                       full barriers count the copies of both CTAs. Allocates
//                       TMEM in both
//   warps 2-9           epilogue: an accumulator's lane is a vocabulary entry,
//                       its column a row; each warp reduces its 32 entries, 32
//                       columns at a time, and merges the candidates into the
//                       rows' 64-bit slots with atomicMax; the accumulator is
//                       released right after the loads, so the next tile's
//                       MMAs overlap the reduction
// Tiles are visited with the rows innermost (tile t: rows t % nm, entries
// t / nm), so the pairs working at one time share weight tiles through L2. A
// second kernel, chained by programmatic dependent launch, turns each slot into
// the index (and the maximum value) and resets it.
//
// What bounds it: few rows the weights' stream, many rows the tensor pipe under
// the power limit and the feed from L2. One CTA per 128 x 256 tile against the
// pairs, us per call (bf16): 48 x 3584 x 152064 172 -> 158 (6.9 TB/s), 128 x
// 4096 x 128256 174 -> 158, 200 rows 200 -> 177, 300 rows 254 -> 221, 854 rows
// 533 -> 504 (1.78 PFLOP/s), 1024 rows 651 -> 570 (1.89), 512 x 4096 x 4096
// 33.6 -> 23.3. In long runs, under the power limit, the 854 rows take 583-593
// instead of 588-595.
// Two blocks per stage: waits, commits and their signals cost a stage about
// 0.28 us whatever it holds (one block: 539 at 854 rows; three, with two stages
// in the ring: 620). Prefetching W towards L2, by the copy unit or by an idle
// warp, made it slower or changed nothing.
//
// Every wait is bounded (2 s); on a timeout the CTA flags DREAMS_DATA_TIMEOUT
// in the status word, merges no further tile, waits for the copies and MMAs it
// issued, meets its peer, whose waits run out likewise, frees its TMEM and exits.
#include <cuda.h>
#include <limits.h>
#include <string.h>

#include <algorithm>

#include "common.cuh"
#include "tc.cuh"
#include "tmap.cuh"

namespace dreams {
namespace {

constexpr int BM = 128;       // vocabulary entries per CTA of a pair
constexpr int MAX_ROWS = 256;  // rows of H per tile
constexpr int BK = 64;         // one 128-byte swizzle row of bf16
constexpr int KB = 2;          // blocks of BK columns per stage
constexpr int MAX_STAGES = 8;
constexpr int LM_THREADS = 320;
constexpr uint32_t A_BLOCK = BM * BK * 2;  // 16 KB
constexpr size_t LM_SMEM = 225 * 1024;     // the ring and its alignment; with the static part within 227 KB

struct LmParams {
  CUtensorMap tmap_h;
  CUtensorMap tmap_w;
  int64_t rows, V;
  int32_t nm, nn, nk;  // tiles along rows and vocabulary; blocks of 64 columns
  unsigned long long *slot;
  int32_t *status;
  uint64_t wait_ns;  // limit of every pipeline wait (2 s unless a test shortens it)
  int32_t stall_at;  // test hook: blocks from this index on (counted per CTA) are never issued (-1: off)
  int32_t n_rows;    // rows of H per tile (a multiple of 32, at most 256)
  int32_t stages;    // of the ring
  uint32_t idesc;    // the MMA's shape
};

// order_key of a valid entry, INT_MIN otherwise, without branches: between the
// warp-wide reductions they cost 131 clk per column.
__device__ __forceinline__ int valid_key(uint32_t u, bool valid) {
  const uint32_t mag = u & 0x7fffffffu;
  int k = int(u ^ (uint32_t(int(u) >> 31) >> 1));
  k = mag == 0u ? 0 : k;
  k = mag > 0x7f800000u ? INT_MAX : k;
  return valid ? k : INT_MIN;
}

__global__ void __launch_bounds__(LM_THREADS, 1) lm_head_argmax_kernel(const __grid_constant__ LmParams P) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_full[MAX_STAGES], bar_empty[MAX_STAGES], bar_tf[2], bar_te[2], bar_never;
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort, s_zero;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();
  // the same offsets in both CTAs (the descriptors hold for both)
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int nk = (P.nk + KB - 1) / KB, n_rows = P.n_rows, stages = P.stages;
  const uint32_t b_block = uint32_t(n_rows) * BK;  // bytes of half the rows, 64 columns
  const uint32_t a_stage = KB * A_BLOCK, b_stage = KB * b_block;
  auto a_s = [&](int st) { return sbase + uint32_t(st) * a_stage; };
  auto b_s = [&](int st) { return sbase + uint32_t(stages) * a_stage + uint32_t(st) * b_stage; };
  const uint32_t full0 = smem_u32(&bar_full[0]), empty0 = smem_u32(&bar_empty[0]);
  const uint32_t tf0 = smem_u32(&bar_tf[0]), te0 = smem_u32(&bar_te[0]);
  if (tid == 0) {
    for (int i = 0; i < stages; ++i) {
      tc::mbar_init(full0 + 8 * i, 1);
      tc::mbar_init(empty0 + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(tf0 + 8 * i, 1);
      tc::mbar_init(te0 + 8 * i, 16);  // one arrival per epilogue warp of the pair
    }
    tc::mbar_init(smem_u32(&bar_never), 1);  // nothing arrives on it (the stall test hook waits on it)
    s_abort = 0;
    s_zero = 0;
    tc::fence_barrier_init();
  }
  if (warp == 1) {
    tc::tmem_alloc_pair(smem_u32(&s_tmem), 512);
    tc::tmem_relinquish_pair();
  }
  tc::fence_before_sync();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers and TMEM are ready
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem;
  grid_wait();
  launch_successor();
  volatile int *abort_flag = &s_abort;
  const uint64_t wait_ns = P.wait_ns;
  auto give_up = [&]() {
    if (*abort_flag == 0) {
      *abort_flag = 1;
      flag(P.status, DREAMS_DATA_TIMEOUT);
    }
  };
  const int64_t ntiles = int64_t(P.nm) * P.nn;
  const int64_t pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;

  if (warp == 0) {
    // ---------------- TMA producer: this CTA's halves of W and H
    if (lane == 0) {
      tc::prefetch_tmap(&P.tmap_h);
      tc::prefetch_tmap(&P.tmap_w);
      const uint32_t pair_bytes = 2 * (a_stage + b_stage);
      const uint32_t lead_full = cluster_addr(&bar_full[0], 0);
      int64_t g = 0;  // stages issued
      int st = 0;     // g % stages
      uint32_t par = 1;  // of the stage's previous use (none in the first round)
      for (int64_t t = pair; t < ntiles && !*abort_flag; t += npairs) {
        const int h0 = int(std::min<int64_t>((t % P.nm) * n_rows + int(rank) * (n_rows / 2), INT_MAX));
        const int w0 = int(t / P.nm) * 2 * BM + int(rank) * BM;
        for (int kb = 0; kb < nk; ++kb, ++g) {
          if (g >= stages && !tc::mbar_wait(empty0 + 8 * st, par, abort_flag, wait_ns)) {
            give_up();
            break;
          }
          if (P.stall_at >= 0 && (g + 1) * KB > P.stall_at) {
            // test hook: these copies are never issued; their consumers' waits
            // run out, like this one on a barrier that nothing arrives on
            tc::mbar_wait(smem_u32(&bar_never), 0, abort_flag, wait_ns);
            give_up();
            break;
          }
          if (rank == 0) tc::mbar_arrive_expect_tx(full0 + 8 * st, pair_bytes);
          // (a last block past the hidden size reads as zeros)
#pragma unroll
          for (int j = 0; j < KB; ++j) {
            const int col = (kb * KB + j) * BK;
            tc::tma_load_2d_pair(a_s(st) + j * A_BLOCK, &P.tmap_w, lead_full + 8 * st, col, w0);
            tc::tma_load_2d_pair(b_s(st) + j * b_block, &P.tmap_h, lead_full + 8 * st, col, h0);
          }
          if (++st == stages) {
            st = 0;
            par ^= 1;
          }
        }
      }
      // no copy may still be landing when the pair ends: the even CTA sees its
      // barriers complete, the odd one its stages consumed
      for (int64_t j = std::max<int64_t>(0, g - stages); j < g; ++j)
        tc::mbar_wait((rank == 0 ? full0 : empty0) + 8 * int(j % stages), (j / stages) & 1, &s_zero, wait_ns);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (the even CTA's)
    if (rank == 0) {
      const uint32_t leader = tc::elect_one();
      const uint32_t idesc = P.idesc;
      const uint64_t ad0 = tc::smem_desc_sw128(a_s(0), 16, 1024);
      const uint64_t bd0 = tc::smem_desc_sw128(b_s(0), 16, 1024);
      int st = 0, it = 0, nd = 0;
      uint32_t par = 0;
      bool ok = true;
      for (int64_t t = pair; t < ntiles && ok; t += npairs, ++it) {
        const int ab = it & 1;
        // the epilogues of both CTAs have read this accumulator's previous tile
        if (it >= 2 && !__all_sync(0xffffffffu, tc::mbar_wait_cluster(te0 + 8 * ab, ((it >> 1) - 1) & 1, abort_flag,
                                                                     wait_ns))) {
          if (leader) give_up();
          break;
        }
        tc::fence_after_sync();
        for (int kb = 0; kb < nk; ++kb) {
          if (!__all_sync(0xffffffffu, tc::mbar_wait(full0 + 8 * st, par, abort_flag, wait_ns))) {
            if (leader) give_up();
            ok = false;
            break;
          }
          tc::fence_after_sync();
#pragma unroll
          for (int k = 0; k < KB * BK / 16; ++k) {  // 16 bf16 along K
            const int j = k / (BK / 16), o = k % (BK / 16) * 32;
            tc::mma_ss_pair(tmem + 256u * ab, ad0 + ((uint32_t(st) * a_stage + j * A_BLOCK + o) >> 4),
                            bd0 + ((uint32_t(st) * b_stage + j * b_block + o) >> 4), idesc,
                            (kb > 0 || k > 0) ? 1u : 0u, leader);
          }
          tc::mma_commit_pair(empty0 + 8 * st, 3, leader);
          if (++st == stages) {
            st = 0;
            par ^= 1;
          }
        }
        // an unfinished tile is announced to this CTA alone, whose epilogue
        // sees the give-up; the other's wait runs out
        __syncwarp();
        tc::mma_commit_pair(tf0 + 8 * ab, ok ? 3 : 1, leader);
        ++nd;
      }
      // every MMA has completed before TMEM is freed
      if (nd > 0) tc::mbar_wait(tf0 + 8 * ((nd - 1) & 1), ((nd - 1) >> 1) & 1, &s_zero);
    }
  } else {
    // ---------------- epilogue warps 2-9: TMEM lane quarter = warp % 4, every
    // second group of 32 columns
    const int q = warp & 3, c0 = warp < 6 ? 0 : 32;
    int it = 0;
    for (int64_t t = pair; t < ntiles; t += npairs, ++it) {
      const int ab = it & 1;
      const int v0 = int(t / P.nm) * 2 * BM + int(rank) * BM + 32 * q;  // this warp's first entry
      const int64_t r0 = (t % P.nm) * n_rows;
      const bool valid = v0 + lane < P.V;
      if (!__all_sync(0xffffffffu, tc::mbar_wait(tf0 + 8 * ab, (it >> 1) & 1, abort_flag, wait_ns))) {
        give_up();
        break;
      }
      if (__any_sync(0xffffffffu, *abort_flag != 0)) break;
      tc::fence_after_sync();
      const uint32_t taddr = tmem + (uint32_t(32 * q) << 16) + 256u * ab;
      // this warp's part of the accumulator is in registers
      auto release = [&]() {
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive_cluster(cluster_addr(&bar_te[ab], 0));
      };
      if (c0 >= n_rows) release();
#pragma unroll 1
      for (int c = c0; c < n_rows; c += 64) {
        uint32_t x[32];
        tc::tmem_ld32(taddr + c, x);
        // slots only grow during the launch: a candidate below is not sent
        const int64_t row = r0 + c + lane;
        const unsigned long long have = row < P.rows ? __ldcg(P.slot + row) : ~0ull;
        tc::tmem_wait_ld();
        if (c + 64 >= n_rows) release();
        // Lane c: column c's greatest key, by exchanges of halves (31 shuffles;
        // a reduction per column took 40 clk each).
#pragma unroll
        for (int e = 0; e < 32; ++e) x[e] = uint32_t(valid_key(x[e], valid));
        int m[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int lo = int(x[e]), hi = int(x[e + 16]);
          m[e] = max((lane & 16) ? hi : lo, __shfl_xor_sync(0xffffffffu, (lane & 16) ? lo : hi, 16));
        }
#pragma unroll
        for (int h = 8; h >= 1; h >>= 1)
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (e < h)
              m[e] = max((lane & h) ? m[e + h] : m[e], __shfl_xor_sync(0xffffffffu, (lane & h) ? m[e] : m[e + h], h));
        const int bk = m[0];
        // its entry only where it may still win (ties go to the lower entry)
        const uint32_t wins = __ballot_sync(0xffffffffu, bk != INT_MIN && pack_key_idx(bk, v0) > have);
        if (wins == 0) continue;
        uint32_t who = 0;
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          const uint32_t at = __ballot_sync(0xffffffffu, int(x[e]) == __shfl_sync(0xffffffffu, bk, e));
          who = lane == e ? at : who;
        }
        if ((wins >> lane) & 1) atomicMax(P.slot + row, pack_key_idx(bk, v0 + __ffs(who) - 1));
      }
    }
  }

  tc::fence_before_sync();
  __syncthreads();
  cluster_sync();  // neither CTA's memory is in use by the other
  if (warp == 1) {
    __syncwarp();
    tc::fence_after_sync();
    tc::tmem_dealloc_pair(tmem, 512);
  }
}

// The row's index (and its maximum value) from its slot; resets the slot. A
// slot that no tile reached (only when a wait gave up: every tile merges a
// candidate, and no (key, index) pair packs to 0) leaves the row untouched.
__global__ void __launch_bounds__(256) lm_head_finish_kernel(unsigned long long *slot, int64_t rows, int32_t *out_idx,
                                                             float *out_max) {
  grid_wait();
  const int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r >= rows) return;
  const unsigned long long v = slot[r];
  if (v == 0ull) return;
  slot[r] = 0ull;
  out_idx[r] = int32_t(~uint32_t(v & 0xffffffffull));
  if (out_max != nullptr) {
    const int key = int(uint32_t(v >> 32) ^ 0x80000000u);
    uint32_t u;
    if (key == INT_MAX) u = 0x7fc00000u;  // NaN
    else if (key >= 0) u = uint32_t(key);
    else u = uint32_t(key ^ 0x7fffffff);
    out_max[r] = __uint_as_float(u);
  }
}

// 2-D view (K innermost, rows) of a row-major bf16 matrix, box (BK, box_rows),
// 128-byte swizzle; rows past the end read as zeros.
bool make_2d_map(CUtensorMap *m, const void *base, int64_t K, int64_t rows, int64_t ld, int box_rows) {
  EncodeTiledFn enc = encode_tiled();
  if (enc == nullptr) return false;
  const cuuint64_t dims[2] = {cuuint64_t(K), cuuint64_t(rows)};
  const cuuint64_t strides[1] = {cuuint64_t(ld) * 2};
  const cuuint32_t box[2] = {cuuint32_t(BK), cuuint32_t(box_rows)};
  const cuuint32_t estr[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace
}  // namespace dreams

using namespace dreams;

extern "C" size_t dreams_lm_head_argmax_workspace_size(int64_t rows) {
  if (rows < 1) return 0;
  return (size_t(rows) * 8 + 255) / 256 * 256;
}

extern "C" dreams_status_t dreams_lm_head_argmax(const void *hidden, int64_t rows, int64_t hidden_dim,
                                                 int64_t ld_hidden, const void *weight, int64_t V, int64_t ld_weight,
                                                 int32_t *out_idx, float *out_max, void *workspace,
                                                 size_t workspace_bytes, int32_t *status_word,
                                                 dreams_stream_t stream) {
  if (hidden == nullptr || weight == nullptr || out_idx == nullptr || rows < 1 || V < 1 || hidden_dim < BK)
    return DREAMS_ERR_INVALID_ARG;
  if (hidden_dim % BK != 0 || ld_hidden < hidden_dim || ld_weight < hidden_dim || ld_hidden % 8 != 0 ||
      ld_weight % 8 != 0 || !aligned16(hidden) || !aligned16(weight) ||
      (out_max != nullptr && (reinterpret_cast<uintptr_t>(out_max) & 3)))
    return DREAMS_ERR_INVALID_ARG;
  if (V > INT_MAX - 2 * BM || rows > (int64_t(1) << 31) || hidden_dim / BK > INT_MAX) return DREAMS_ERR_UNSUPPORTED;
  if (workspace == nullptr || workspace_bytes < dreams_lm_head_argmax_workspace_size(rows) || !aligned16(workspace))
    return DREAMS_ERR_WORKSPACE;
  LmParams P;
  memset(&P, 0, sizeof(P));
  // The tile's height: the fewest rounds over the pairs, weighted by what a
  // block costs each SM to load. (512 x 4096 x 4096: 128 rows per tile 23.3 us,
  // 256, which leave most pairs idle, 36.3.)
  const int64_t npairs = std::max(1, num_sms() / 2), nn = (V + 2 * BM - 1) / (2 * BM);
  const int64_t fewest = (rows + MAX_ROWS - 1) / MAX_ROWS;
  int64_t nm = 0, best = INT64_MAX;
  int n_rows = 0;
  for (int64_t m = fewest; m < fewest + 8; ++m) {
    const int64_t n = ((rows + m - 1) / m + 31) / 32 * 32, tiles = (rows + n - 1) / n;
    const int64_t cost = (tiles * nn + npairs - 1) / npairs * (BM + n / 2);
    if (cost < best) {
      best = cost;
      nm = tiles;
      n_rows = int(n);
    }
  }
  if (!make_2d_map(&P.tmap_h, hidden, hidden_dim, rows, ld_hidden, n_rows / 2) ||
      !make_2d_map(&P.tmap_w, weight, hidden_dim, V, ld_weight, BM))
    return DREAMS_ERR_UNSUPPORTED;
  P.rows = rows;
  P.V = V;
  P.nm = int32_t(nm);
  P.nn = int32_t(nn);
  P.n_rows = n_rows;
  P.stages = int32_t(std::min<size_t>(MAX_STAGES, (LM_SMEM - 1024) / (KB * (A_BLOCK + size_t(n_rows) * BK))));
  P.idesc = tc::idesc_bf16_f32(2 * BM, n_rows, false);
  P.nk = int32_t(hidden_dim / BK);
  P.slot = static_cast<unsigned long long *>(workspace);
  P.status = status_word;
  test_stall(DREAMS_TEST_LM_HEAD, &P.stall_at, &P.wait_ns);
  dreams_status_t st = ensure_max_dynamic_smem(reinterpret_cast<const void *>(lm_head_argmax_kernel), int(LM_SMEM));
  if (st != DREAMS_OK) return st;
  const unsigned grid = unsigned(2 * std::min(nm * nn, npairs));
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  st = launch_clusters(lm_head_argmax_kernel, dim3(grid), dim3(LM_THREADS), LM_SMEM, s, 2, P);
  if (st != DREAMS_OK) return st;
  return launch_kernel(lm_head_finish_kernel, dim3(unsigned((rows + 255) / 256)), dim3(256), 0, s, P.slot, rows, out_idx,
                       out_max);
}
