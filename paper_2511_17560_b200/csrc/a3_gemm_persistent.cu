// Persistent CTA-pair GEMMs of the recompute path (the feed-forward part of H(.) in Eq. 5) with the operand roles
// swapped:   SwiGLU    out[t][f] = silu(x[t] . Wg[f]) * (x[t] . Wu[f])
//            residual  C[t][f] += x[t] . W[f]            (output projection, MLP down projection)
//
// Why another kernel.  With one CTA per 128-token x 256-column tile an SM pulls 48 KiB per k-block through its L2
// port and that, not the tensor pipe, sets the pace (a wave's time follows the bytes: about 107 GB/s per SM with
// 192 KiB in flight); at 804 tokens the 128-row tiles also pad the rows to 896 and the grid to three waves.  Here
//   * the WEIGHTS are the M-side operand of tcgen05.mma.cta_group::2 (M = 256 over a CTA pair).  SwiGLU: each CTA
//     holds 64 gate rows and 64 up rows of the same 64 features (its 128 accumulator lanes), so gate and up of a
//     feature meet inside one CTA; residual: 128 rows of the one matrix;
//   * the TOKENS are the N-side operand, in tiles of N <= 256 tokens chosen to divide the row count evenly
//     (804 rows -> 4 x 208: 3 % padding instead of 11 %); each CTA loads half of the token tile, the instruction
//     reads both halves.  Per k-block an SM pulls 16 KiB of weights + N/2 token rows (13 KiB at N = 208);
//   * the kernel is persistent: CTA pair p walks units p, p + pairs, ... (unit = 128 (SwiGLU) or 256 features x one
//     token tile), accumulators are double-buffered in tensor memory (2 x N <= 512 columns), so the epilogue of a
//     unit runs under the main loop of the next one; a ring stage holds two k-blocks (one barrier hand-shake and one
//     commit per eight instructions: the single issuing thread, not the pipe, was the limit with one).
// Epilogues: accumulator lanes are features, so values go through shared memory once, where gate meets up and a rotation
// pair its other half, and leave token by token in 16-byte stores.  Measured at Llama-8B width: tensor pipe 97 % active at
// 5 152 rows.
// No load uses cluster multicast.  Every wait is bounded (see a3_tc.cuh): a waiter that gives up raises the CTA's
// abort flag and the device status bit, all roles leave their loops, tensor memory is released and the CTA returns.
#include <cuda.h>

#include <type_traits>

#include "a3_internal.cuh"
#include "a3_tc.cuh"

namespace a3 {

constexpr int SP_THREADS = 320;  // warp 0: TMA, warp 1: MMA (leader CTA), warps 2..9: epilogue (two sets of four)
constexpr int SP_MAX_STAGES = 8;
constexpr int SP_SUB = 2;  // k-blocks of 64 per ring stage: one barrier hand-shake and one commit per 8 MMAs
constexpr int SP_FEAT = 64;                              // features per CTA (64 gate lanes + 64 up lanes)
constexpr int SP_A_BYTES = 2 * SP_FEAT * TC_BK * 2;      // 16 KiB: gate rows, then up rows
// Exchange buffers of the epilogues, which take `chunk` tokens at a time (32 where that costs no ring stage, else 16 or 8: see
// set_stages): per warp set four quarters of [chunk][32 lanes] fp32, 16 bytes apart in the banks.
__host__ __device__ constexpr int sp_set_floats(int chunk) { return 4 * (chunk * 32 + 4); }
// both sets, 256-byte aligned, and for QKV the checked positions of each set's tokens behind them
__host__ __device__ constexpr int sp_xch_floats_bytes(int chunk) { return (2 * sp_set_floats(chunk) * 4 + 255) & ~255; }
__host__ __device__ constexpr int sp_xch_bytes(int epi, int chunk) { return sp_xch_floats_bytes(chunk) + (epi == EPI_QKV ? 1024 : 0); }
constexpr int SP_SMEM_LIMIT = 227 * 1024;
constexpr int SP_SLOTS = 3;  // accumulators in tensor memory, at most

struct SpParams {
  int M, K, F;
  int tok_tiles, tok_n;  // token tiles of a launch (TT > 1: groups of TT) and tokens per tile (multiple of 16, at most 256)
  int n_fblocks;         // feature blocks (one per CTA pair and unit): units = n_fblocks x tok_tiles
  int group;             // feature blocks per group of the unit order (1: feature blocks outermost)
  int early;             // the first ring stages' weights may be loaded before the preceding kernels are waited for
  int k_slices;          // SPLIT: slices of the k-loop per (feature block, token tile); 1 otherwise
  float* part;           // SPLIT: fp32 partial sums [k_slices][M][F]
  int n_units, n_pairs;
  int stages, stage_bytes;  // ring depth; bytes per stage: SP_SUB / TT k-blocks of weights, then as many of this CTA's half of every token tile
  int slot_cols;         // tensor-memory columns from one accumulator to the next
  int chunk;             // tokens per exchange of the epilogue: 32, 16 or (not QKV) 8
  bf16* C;
  int ldc;
  uint32_t* status;
  // EPI_QKV: the concatenated heads of up to three matrices (q, k, v in any subset), 128 features each
  int n_heads;
  int seg_heads_end[3];  // cumulative head counts of the segments
  int kind[3];           // 0 = q, 1 = k, 2 = v
  const bf16* bias[3];
  bf16 *q_out, *k_cache, *v_cache;
  const int32_t* pos;
  int kv_len, Hq, Hkv, layout, max_pos;
  const float2* tab;
  // queries of the rows from q_first on only (the matrices are k, v, q in this order): units from q_unit0 on are head pairs from
  // q_block0 on x q_tiles token tiles that start at row q_first.  Otherwise q_unit0 = n_units, q_first = 0.
  int q_first, q_unit0, q_block0, q_tiles;
};

__device__ __forceinline__ void named_bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// arrives on the barrier at the same shared-memory offset in CTA `cta` of the cluster
__device__ __forceinline__ void mbar_arrive_in_cta(uint32_t bar, uint32_t cta) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(bar), "r"(cta));
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}
// w (8 .. CH in steps of 8; uniform for the warp) consecutive accumulator columns of this thread's lane
template <int CH>
__device__ __forceinline__ void sp_ld_chunk(uint32_t taddr, int w, float* v) {
  if (CH == 32 && w == 32) {
    tc_ld32(taddr, v);
  } else {  // static register indices: the array must not go to local memory
#pragma unroll
    for (int i = 0; i < CH / 8; ++i)
      if (w >= 8 * i + 8) tc_ld8(taddr + 8 * i, v + 8 * i);
  }
  tc_wait_ld_of<CH>(v);
}
// 32 bytes (aligned to 32) through the read-only path.  The lanes of a token read its table row 64 bytes apart, so that a load costs
// its lines and not its bytes: half as many loads.  A chunk's fetch took 800 of its 1 450 clocks; request of 369 tokens on a small
// model 144.1 -> 142.8 us (a prefill of 512 tokens at Llama-8B width does not show it: 0.25 % where two runs differ by 0.8).
__device__ __forceinline__ void ldg32(const float4* p, float4& a, float4& b) {
  asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
               : "l"(p));
}
// f(std::integral_constant<int, chunk>) for the chunk of this launch
template <bool MAY_8, typename F>
__device__ __forceinline__ bool sp_with_chunk(int chunk, F f) {
  if (chunk == 32) return f(std::integral_constant<int, 32>());
  if constexpr (MAY_8) {
    if (chunk == 8) return f(std::integral_constant<int, 8>());
  }
  return f(std::integral_constant<int, 16>());
}

// Stores of the first `valid` of CH tokens, eight at a time without a branch in between: a branch around every store makes
// a block of its own of every token's arithmetic, and its latency (exchange, exponential, reciprocal: 160 clocks) was paid
// token by token - 5 000 clocks for the 32 of a chunk.
template <int CH, typename F>
__device__ __forceinline__ void sp_store_tokens(int valid, F store) {
#pragma unroll
  for (int i = 0; i < CH; i += 8) {
    if (valid >= i + 8) {
#pragma unroll
      for (int e = i; e < i + 8; ++e) store(e);
    } else {
#pragma unroll
      for (int e = i; e < i + 8; ++e)
        if (e < valid) store(e);
    }
  }
}

// Unit u -> (feature block, token tile).  Units are numbered in groups of `group` feature blocks, token tiles next,
// the group's blocks innermost.  With group = 8 the 74 pairs that work side by side cover about 8 feature blocks x 9
// token tiles, and since they walk the k-blocks at the same pace, what a round pulls through L2 is 8 weight blocks +
// 9 token tiles: the order for token matrices that do not fit in L2 (with feature blocks outermost a round of the
// 32 800-row QKV launch pulled 1 weight block + 74 token tiles: 6.9 GB of DRAM reads for 0.3 GB of operands).  With
// group = 1 (feature blocks outermost) every round walks all token tiles: the order for token matrices that stay in
// L2, where the weights then stream through exactly once (SwiGLU at 5 152 rows: 418 MB of DRAM reads against 719 MB
// with groups of 8).
__device__ __forceinline__ void sp_unit(int u, int n_fblocks, int tok_tiles, int group, int& fb, int& tt) {
  const int per_group = group * tok_tiles;
  const int g = u / per_group, r = u - g * per_group;
  const int gsz = min(group, n_fblocks - g * group);
  tt = r / gsz;
  fb = g * group + (r - tt * gsz);
}

// The same with the first row of the token tile, QKV units of late queries included (see SpParams)
template <int EPI>
__device__ __forceinline__ void sp_place(const SpParams& p, int u, int& fb, int& row0) {
  int tt;
  if (EPI == EPI_QKV && u >= p.q_unit0) {
    fb = p.q_block0 + (u - p.q_unit0) / p.q_tiles;
    row0 = p.q_first + (u - p.q_unit0) % p.q_tiles * p.tok_n;
    return;
  }
  sp_unit(u, p.n_fblocks, p.tok_tiles, p.group, fb, tt);
  row0 = tt * p.tok_n;
}

// Ring stages [first, first + count) of slice ks of a k-loop of kt k-blocks.  The cuts lie between groups of SP_SUB k-blocks whatever a
// stage holds (SP_SUB / TT of them), so that the partial sums of a slice do not depend on how many token tiles share its weights.
template <int TT>
__device__ __forceinline__ void sp_slice(int ks, int k_slices, int kt, int& first, int& count) {
  const long long groups = kt / SP_SUB;
  const int g0 = (int)(groups * ks / k_slices);
  first = g0 * TT;
  count = ((int)(groups * (ks + 1) / k_slices) - g0) * TT;
}

// D += A B over the CTA pair (accumulating form: no predicate to set up)
__device__ __forceinline__ void tc_mma_pair_acc(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.eq.u32 p, 0, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc)
      : "memory");
}

// EPI_SWIGLU: tmG/tmU are the gate and up matrices (box of 64 rows each); EPI_RESIDUAL: tmG is the one weight matrix
// (box of 128 rows, tmU unused) and the epilogue adds the accumulator to C in place.
// EPI_QKV: tmG / tmU / tmW are the matrices of the segments (boxes of 128 rows: one head); a unit is two consecutive
// heads of the concatenated list, one per CTA of the pair, times one token tile; the epilogue adds the bias, rotates
// q and k at the tokens' positions (the two halves of a rotation pair sit 64 lanes apart and meet through shared
// memory, like gate and up) and writes q to its buffer and k, v into the cache rows pos[token] (the scatter of Eq. 5).
// SPLIT: a launch with fewer units than CTA pairs cuts the k-loop of every unit into k_slices and the epilogue writes
// the slice's fp32 sums to `part` instead; the kernel that follows (RMSNorm, which reads these rows anyway) adds the
// slices in order.  See residual_slices below for when and why.
// KC = 2 (QKV of few rows): a cluster of two pairs per unit, each with half of the k-loop.  The epilogue needs whole sums: pair c
// finishes the tokens of warp set c and receives the other pair's sums for them through distributed shared memory.
// ONCE: every weight is read once and leaves L2 first (see weights_once and the producer).
// TT = 2 (just over 256 rows): a unit is two token tiles on one stream of weights, see two_tiles.  A ring stage is then one k-block:
// eight instructions again.  Accumulators take turns in three slots of tensor memory instead of two.
template <int EPI, bool SPLIT, int KC, bool ONCE, int TT = 1>
__global__ void __cluster_dims__(2 * KC, 1, 1) __launch_bounds__(SP_THREADS, 1)
pair_t_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmG,
              const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmW, const SpParams p) {
  constexpr int ROWS = EPI == EPI_SWIGLU ? SP_FEAT : 2 * SP_FEAT;  // output features per CTA
  constexpr int SUB = SP_SUB / TT;          // k-blocks per ring stage
  constexpr int SLOTS = TT == 1 ? 2 : SP_SLOTS;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t base = smem_u32(smem_raw);  // same offset in both CTAs of the pair
  unsigned char* base_ptr = smem_raw;
  if (base & 1023u) {  // the swizzled tiles need a 1024-byte aligned window; uniform for the launch, nothing is set up yet
    if (threadIdx.x == 0) atomicOr(p.status, A3_DEV_WAIT_EXHAUSTED);
    return;
  }
  const int S = p.stages;
  const int xch_off = S * p.stage_bytes, bar_off = xch_off + (SPLIT ? 0 : sp_xch_bytes(EPI, p.chunk));
  // barriers (8 bytes each): full[8] (used in the leader), empty[8], tmem_full[3], tmem_empty[3] (used in the leader)
  const uint32_t bars = base + bar_off;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (SP_MAX_STAGES + s); };
  auto tmem_full = [&](int b) { return bars + 8u * (2 * SP_MAX_STAGES + b); };
  auto tmem_empty = [&](int b) { return bars + 8u * (2 * SP_MAX_STAGES + SP_SLOTS + b); };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(base_ptr + bar_off + 8 * (2 * SP_MAX_STAGES + 2 * SP_SLOTS));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + bar_off + 8 * (2 * SP_MAX_STAGES + 2 * SP_SLOTS) + 8);
  volatile int* ep_ok = abort_flag + 2;  // the epilogue's one waiter tells the other 127 threads how its wait ended
  float* xch = reinterpret_cast<float*>(base_ptr + xch_off);

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const uint32_t crank = cluster_ctarank(), rank = crank & 1u;  // CTA of the cluster, CTA of the pair
  const int kc = (int)(crank >> 1);                             // the pair's part of the k-loop (KC > 1)
  const uint32_t pair_cta0 = crank & ~1u;
  const uint16_t pair_mask = (uint16_t)(3u << pair_cta0);
  const bool leader = rank == 0;
  const int pair = blockIdx.x / (2 * KC);
  int merged = 0;  // KC > 1: how many of the two cluster barriers of the merge this warp has passed
  const int KT = p.K / TC_BK, KS = KT / SUB;  // k-blocks (a multiple of SP_SUB, checked by the launcher) and ring stages of a k-loop
  const int half_n = p.tok_n >> 1;  // token rows this CTA loads per k-block (multiple of 8)
  const uint32_t b_bytes = (uint32_t)half_n * TC_BK * 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < SLOTS; ++b) {
      mbar_init(tmem_full(b), 1);
      mbar_init(tmem_empty(b), 16);  // every epilogue warp of both CTAs
    }
    abort_flag[0] = 0;
    abort_flag[1] = 0;
    ep_ok[0] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {  // the same warp of both CTAs
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cluster_sync_all();  // the peer's barriers exist before anything is signalled on them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // The weights are nobody's output: the producer fills the ring's weight half before it waits for the preceding kernel
  // (16 KiB x 2 per stage and CTA, most of what a launch of few rows spends its first microseconds on); everybody else
  // waits here.
  if (warp != 0 || !p.early) {
    pdl_wait();
    pdl_launch_dependents();  // from here on: a launch never runs ahead of more than the one before it
  }

  // Accumulators of this pair, numbered in order: number t lies in slot t % SLOTS.  It goes back to the MMA issuer, which takes the slot
  // again SLOTS accumulators later.  Behind the last ones nobody waits, and an arrival still on its way must not find the leader
  // gone (the last barrier orders no memory).
  const int n_acc = pair < p.n_units ? TT * ((p.n_units - pair + p.n_pairs - 1) / p.n_pairs) : 0;
  auto awaited = [&](int t) { return t + SLOTS < n_acc; };
  // An epilogue that gives a wait up may have sent arrivals that the issuer, which has given up as well, never took.  (Every epilogue
  // with such an arrival gives up: the accumulator that would have been computed in that slot, for which it waits, is never published.)
  // Its fence and the last barrier order them before the leader goes.
  auto give_up = [] { asm volatile("fence.acq_rel.cluster;" ::: "memory"); };
  if (warp == 0) {
    // ---------------- TMA producer (both CTAs): own gate/up rows, own half of the token tile
    // as a whole warp, one elected lane issuing; a stage's k-blocks of an operand are one copy of a 3-D map ([k-block][row][64])
    {
      if (elect_one()) {
        tmap_prefetch(&tmX);
        tmap_prefetch(&tmG);
        if (EPI != EPI_RESIDUAL) tmap_prefetch(&tmU);
        if (EPI == EPI_QKV) tmap_prefetch(&tmW);
      }
      // ONCE (see weights_once): first out, so that they do not displace what the kernels hand on (rows, partial sums, the
      // cache) and their code.  A layer of 144 rows at Llama-8B width 115.6 -> 111.7 us, of 75 rows at Qwen-7B width 91.3 -> 89.6.
      // With two token tiles a policy on every load costs (280 rows 138.1 -> 140.5), and so does choosing per load (270 rows,
      // Qwen width 122.7 -> 123.6): hence an instance of its own.
      const uint64_t once = ONCE ? l2_evict_first() : 0;
      auto load = [&](uint32_t dst, const CUtensorMap* map, int y, int z, uint32_t bar) {
        if (ONCE) tma_load_3d_pair_once(dst, map, y, z, bar, once);
        else tma_load_3d_pair(dst, map, y, z, bar);
      };
      int kbg = 0, issued = 0;
      int s = 0;        // ring position and phase, kept by counting: S is a run-time value and a division per
      uint32_t ph = 0;  // k-block is a long dependent chain in a one-thread role
      bool ok = true;
      int early = p.early ? S : 0;  // ring stages whose weights are requested ahead of pdl_wait (within the first unit)
      for (int u = pair; u < p.n_units && ok; u += p.n_pairs) {
        int fb, row0, kb0 = 0, kb1 = KT;
        sp_place<EPI>(p, SPLIT ? u / p.k_slices : u, fb, row0);
        if (SPLIT) {
          sp_slice<TT>(u % p.k_slices, p.k_slices, KT, kb0, kb1);
          kb0 *= SUB;
          kb1 = kb0 + kb1 * SUB;
        } else if (KC > 1) {
          sp_slice<TT>(kc, KC, KT, kb0, kb1);
          kb0 *= SUB;
          kb1 = kb0 + kb1 * SUB;
        }
        int f0 = fb * (2 * ROWS) + (int)rank * ROWS;
        const CUtensorMap* mapA = &tmG;
        if (EPI == EPI_QKV) {
          // this CTA's head of the concatenated list -> its matrix and first row there (a pair beyond the last head of
          // an odd list loads head 0 again; its epilogue stores nothing)
          int hd = 2 * fb + (int)rank;
          if (hd >= p.n_heads) hd = 0;
          const int sg = (hd >= p.seg_heads_end[0]) + (hd >= p.seg_heads_end[1]);
          f0 = (hd - (sg == 0 ? 0 : p.seg_heads_end[sg - 1])) * 128;
          mapA = sg == 0 ? &tmG : (sg == 1 ? &tmU : &tmW);
        }
        const int t0 = row0 + (int)rank * half_n;
        auto load_weights = [&](int stage, int kb) {
          const uint32_t full_leader = full_bar(stage) & PAIR_LEADER_MASK, sa = base + stage * p.stage_bytes;
          // the leader announces the bytes of both CTAs; a copy of the peer that completes earlier cannot end the
          // phase, because the leader's own arrival is still pending until its expect_tx
          if (elect_one()) {
            if (leader) mbar_expect_tx(full_bar(stage), 2 * SUB * (SP_A_BYTES + TT * b_bytes));
            if (EPI == EPI_SWIGLU) {
              // a k-block's operand is gate rows, then up rows
#pragma unroll
              for (int j = 0; j < SUB; ++j) {
                load(sa + j * SP_A_BYTES, &tmG, f0, kb + j, full_leader);
                load(sa + j * SP_A_BYTES + SP_A_BYTES / 2, &tmU, f0, kb + j, full_leader);
              }
            } else {
              load(sa, mapA, f0, kb, full_leader);
            }
          }
          __syncwarp();
        };
        if (early && kbg == 0) {
          early = min(early, (kb1 - kb0) / SUB);
          for (int i = 0; i < early; ++i) load_weights(i, kb0 + i * SUB);
          issued = early;
          pdl_wait();
          pdl_launch_dependents();
        }
        for (int kb = kb0; kb < kb1; kb += SUB, ++kbg) {
          if (kbg >= early) {
            if (!mbar_wait_warp(empty_bar(s), ph ^ 1, abort_flag, p.status)) {
              ok = false;
              break;
            }
            load_weights(s, kb);
          }
          if (elect_one()) {
#pragma unroll
            for (int j = 0; j < TT; ++j)
              tma_load_3d_pair(base + s * p.stage_bytes + SUB * (SP_A_BYTES + j * b_bytes), &tmX, t0 + j * p.tok_n, kb, full_bar(s) & PAIR_LEADER_MASK);
          }
          __syncwarp();
          issued = max(issued, kbg + 1);
          if (++s == S) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (lane == 0 && *abort_flag) {
        // let the copies already issued land before the CTA can exit (bounded)
        if (leader) {
          for (int k = max(0, issued - S); k < issued; ++k)
            mbar_wait(full_bar(k % S), (k / S) & 1, abort_flag + 1, p.status, 2000000ull);
        } else {
          const unsigned long long t0 = global_ns();
          while (global_ns() - t0 < 200000ull) {
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: the leader alone, for both CTAs.
    // The whole warp walks the loop, one elected lane issues (see uniform_warp).  Back to back at 804 rows x
    // 28 672 columns 167 -> 156 us, at 133 rows 54.3 -> 51.1, a single unit alone (no contention) 19.7 -> 16.0.
    if (leader) {
      const uint32_t idesc = idesc_bf16_pair(p.tok_n);
      const uint64_t da0 = smem_desc_sw128(base), db0 = smem_desc_sw128(base + SUB * SP_A_BYTES);
      // descriptor address fields count 16-byte units: stage and k-step offsets are added to the first stage's
      const uint32_t stage16 = (uint32_t)p.stage_bytes >> 4, a_sub16 = SP_A_BYTES >> 4, b_sub16 = (uint32_t)half_n * (TC_BK * 2) >> 4;
      const uint32_t tmem_acc = __shfl_sync(0xffffffffu, tmem_base, 0);
      int per_unit = KS, total = 0;
      if (KC > 1) {
        int first;
        sp_slice<TT>(kc, KC, KT, first, per_unit);
      }
      if (SPLIT) {
        for (int u = pair, first; u < p.n_units; u += p.n_pairs) {
          int count;
          sp_slice<TT>(u % p.k_slices, p.k_slices, KT, first, count);
          total += count;
        }
      } else {
        total = n_acc / TT * per_unit;
      }
      int s = 0, u = pair, in_unit = 0, slot[TT];
      uint32_t ph = 0, stage_off = 0, slot_ph = 1, d[TT];  // slot: of the next accumulator, phase in which it is found empty
      int next_slot = 0;
      bool ok = total > 0;
      for (int g = 0; g < total && ok; ++g) {
        if (in_unit == 0) {
#pragma unroll
          for (int j = 0; j < TT; ++j) {
            // the epilogues of both CTAs have drained this accumulator (first use: passes at once)
            slot[j] = next_slot;
            ok = ok && mbar_wait_warp(tmem_empty(next_slot), slot_ph, abort_flag, p.status);
            d[j] = tmem_acc + (uint32_t)(next_slot * p.slot_cols);
            if (++next_slot == SLOTS) {
              next_slot = 0;
              slot_ph ^= 1;
            }
          }
          if (!ok) break;
          if (SPLIT) {
            int first;
            sp_slice<TT>(u % p.k_slices, p.k_slices, KT, first, per_unit);
          }
        }
        ok = mbar_wait_warp(full_bar(s), ph, abort_flag, p.status);
        if (!ok) break;
        tc_fence_after();
        const uint64_t da_s = da0 + stage_off, db_s = db0 + stage_off;
        if (elect_one()) {
#pragma unroll
          for (int j = 0; j < TT; ++j) {
            const uint64_t db_j = db_s + (uint64_t)(j * SUB * b_sub16);
            tc_mma_pair_f16(d[j], da_s, db_j, idesc, in_unit != 0);
#pragma unroll
            for (int i = 1; i < SUB * (TC_BK / 16); ++i) {
              const int b = i / (TC_BK / 16), k = i % (TC_BK / 16);
              tc_mma_pair_acc(d[j], da_s + (uint64_t)(b * a_sub16 + 2 * k), db_j + (uint64_t)(b * b_sub16 + 2 * k), idesc);
            }
          }
          tc_commit_pair(empty_bar(s), pair_mask);  // frees this stage in both CTAs once the instructions above have read it
          if (in_unit + 1 == per_unit) {
#pragma unroll
            for (int j = 0; j < TT; ++j) tc_commit_pair(tmem_full(slot[j]), pair_mask);  // publishes the accumulators in both CTAs
          }
        }
        __syncwarp();
        if (++in_unit == per_unit) {
          in_unit = 0;
          u += p.n_pairs;
        }
        stage_off += stage16;
        if (++s == S) {
          s = 0;
          ph ^= 1;
          stage_off = 0;
        }
      }
    }
  } else if (SPLIT) {
    // ---------------- epilogue of a k-slice: warps 2..9 of both CTAs, lane = feature (of the one matrix or of this CTA's
    // head), warp set 0 the first half of the token columns, set 1 the second; a warp writes 32 consecutive fp32 sums of
    // one token (128 bytes) per instruction.
    const int quarter = warp & 3;
    const int set = (warp - 2) >> 2;
    const int ep_tid = (warp - 2) * 32 + lane;
    const int set_n = p.tok_n >> 1;
    const int n_chunks = (set_n + 31) >> 5;
    int b = 0;
    uint32_t b_ph = 0;
    for (int t = 0; t < n_acc; ++t) {
      const int u = pair + t / TT * p.n_pairs;
      int fb, tt;
      sp_unit(u / p.k_slices, p.n_fblocks, p.tok_tiles, p.group, fb, tt);
      const int f = fb * (2 * ROWS) + (int)rank * ROWS + quarter * 32 + lane;
      const int t0 = (tt * TT + t % TT) * p.tok_n + set * set_n;
      float* prow = p.part + ((size_t)(u % p.k_slices) * p.M + t0) * p.F + f;
      if (ep_tid == 0) ep_ok[0] = mbar_wait(tmem_full(b), b_ph, abort_flag, p.status) ? 1 : 0;
      named_bar_sync(1, 256);
      if (!ep_ok[0]) {  // uniform for the 256 threads
        give_up();
        break;
      }
      tc_fence_after();
      const uint32_t trow = tmem_base + (uint32_t)(b * p.slot_cols) + (uint32_t)(set * set_n) + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
      for (int c = 0; c < n_chunks; ++c) {
        const int w = min(32, set_n - c * 32);
        float v[32];
        __syncwarp();
        sp_ld_chunk<32>(trow + c * 32, w, v);
        const int valid = f < p.F ? min(w, p.M - (t0 + c * 32)) : 0;
        float* pc = prow + (size_t)(c * 32) * p.F;
        sp_store_tokens<32>(valid, [&](int e) { pc[(size_t)e * p.F] = v[e]; });
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0 && awaited(t)) mbar_arrive_in_cta(tmem_empty(b), pair_cta0);
      if (++b == SLOTS) {
        b = 0;
        b_ph ^= 1;
      }
    }
  } else if (EPI == EPI_SWIGLU) {
    // ---------------- epilogue, silu(gate) * up: warps 2..9 of both CTAs; warp w may touch TMEM lanes 32*(w%4) .. +31: lanes
    // 0..63 hold the gate rows of this CTA's 64 features, lanes 64..127 their up rows.  Warp set 0 (warps 2..5) takes the
    // first half of the token columns, set 1 (warps 6..9) the second, a chunk at a time in two phases as in the QKV
    // epilogue: feature-major out of tensor memory into shared memory, then token-major, a thread taking 8 features of a
    // token: their gates, their ups and one 16-byte store.
    const int quarter = warp & 3;
    const int set = (warp - 2) >> 2;
    const int ep_tid = (warp - 2) * 32 + lane;
    const int st = quarter * 32 + lane;  // thread within the set
    const int set_n = p.tok_n >> 1;      // token columns of a set (multiple of 8)
    const int bar_set = 2 + set;
    sp_with_chunk<true>(p.chunk, [&](auto chunk) {
      constexpr int CH = decltype(chunk)::value, QUARTER = CH * 32 + 4, PASSES = (CH + 15) / 16;
      const int n_chunks = (set_n + CH - 1) / CH;
      float* xset = xch + set * sp_set_floats(CH);
      float* xmine = xset + quarter * QUARTER + lane;
      // phase 2 assignment: token e2 (+ 16 per pass; half of the threads idle in chunks of 8), features 8 (st & 7) .. + 7
      const int e2 = st >> 3, fg = st & 7;
      const float* xg = xset + (fg >> 2) * QUARTER + (fg & 3) * 8;
      const float* xu = xg + 2 * QUARTER;
      int b = 0;
      uint32_t b_ph = 0;
      for (int t = 0; t < n_acc; ++t) {
        int fb, tt;
        sp_unit(pair + t / TT * p.n_pairs, p.n_fblocks, p.tok_tiles, p.group, fb, tt);
        const int t0 = (tt * TT + t % TT) * p.tok_n + set * set_n;
        const int valid = min(set_n, p.M - t0);  // tokens of this set that exist (may be <= 0)
        bf16* out = p.C + (size_t)max(t0, 0) * p.ldc + fb * (2 * SP_FEAT) + (int)rank * SP_FEAT + fg * 8;
        if (ep_tid == 0) ep_ok[0] = mbar_wait(tmem_full(b), b_ph, abort_flag, p.status) ? 1 : 0;
        named_bar_sync(1, 256);
        if (!ep_ok[0]) {  // uniform for the 256 threads
          give_up();
          return false;
        }
        tc_fence_after();
        const uint32_t trow = tmem_base + (uint32_t)(b * p.slot_cols) + (uint32_t)(set * set_n) + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
        for (int c = 0; c < n_chunks; ++c) {
          float v[CH];
          __syncwarp();
          sp_ld_chunk<CH>(trow + c * CH, min(CH, set_n - c * CH), v);
#pragma unroll
          for (int e = 0; e < CH; ++e) xmine[e * 32] = v[e];
          named_bar_sync(bar_set, 128);
          uint4 r[PASSES];
#pragma unroll
          for (int pass = 0; pass < PASSES; ++pass) {
            const int e = min(e2 + 16 * pass, CH - 1);
            float g[8], up[8];
            *reinterpret_cast<float4*>(g) = *reinterpret_cast<const float4*>(xg + e * 32);
            *reinterpret_cast<float4*>(g + 4) = *reinterpret_cast<const float4*>(xg + e * 32 + 4);
            *reinterpret_cast<float4*>(up) = *reinterpret_cast<const float4*>(xu + e * 32);
            *reinterpret_cast<float4*>(up + 4) = *reinterpret_cast<const float4*>(xu + e * 32 + 4);
#pragma unroll
            for (int k = 0; k < 8; ++k) g[k] = silu_mul(g[k], up[k]);
            r[pass] = pack8(g);
          }
#pragma unroll
          for (int pass = 0; pass < PASSES; ++pass) {
            const int e = e2 + 16 * pass;
            if (e < CH && c * CH + e < valid) *reinterpret_cast<uint4*>(out + (size_t)(c * CH + e) * p.ldc) = r[pass];
          }
          named_bar_sync(bar_set, 128);  // everybody has read this chunk's values
        }
        // this warp has read its part of the accumulator (wait::ld in sp_ld_chunk): it goes back to the MMA issuer
        tc_fence_before();
        __syncwarp();
        if (lane == 0 && awaited(t)) mbar_arrive_in_cta(tmem_empty(b), pair_cta0);
        if (++b == SLOTS) {
          b = 0;
          b_ph ^= 1;
        }
      }
      return true;
    });
  } else if (EPI == EPI_QKV) {
    // ---------------- epilogue, q / k / v heads: warps 2..9 of both CTAs; warp w may touch TMEM lanes 32*(w%4) .. +31,
    // lane = feature of this CTA's head; warp set 0 (warps 2..5) takes the first half of the token columns, set 1 the
    // second.  While the unit's main loop runs, the set fetches and checks the positions of its tokens and the table rows
    // of its first chunk.  Then a chunk of tokens at a time, in two phases around a named barrier of the set's 128 threads:
    //   1. feature-major: every warp reads its 32 features x chunk from tensor memory, adds the bias and parks the
    //      values in shared memory;
    //   2. token-major: a thread takes 8 consecutive features of the head's first half and the 8 that lie 64 further of
    //      ONE token (both halves of its rotation pairs, whichever the pairing), rotates them with the token's table row,
    //      fetched a chunk ahead in 16-byte loads, and writes two 16-byte vectors: a warp stores 512 contiguous-by-row
    //      bytes per instruction where a lane-per-feature epilogue stores 64.
    const int quarter = warp & 3;
    const int set = (warp - 2) >> 2;
    const int ep_tid = (warp - 2) * 32 + lane;
    const int st = quarter * 32 + lane;  // thread within the set
    const int set_n = p.tok_n >> 1;
    const int bar_set = 2 + set;
    sp_with_chunk<false>(p.chunk, [&](auto chunk) {
      constexpr int CH = decltype(chunk)::value, QUARTER = CH * 32 + 4, PASSES = CH / 16;
      const int n_chunks = (set_n + CH - 1) / CH;
      float* xset = xch + set * sp_set_floats(CH);
      int* posbuf = reinterpret_cast<int*>(base_ptr + xch_off + sp_xch_floats_bytes(CH)) + set * 128;
      // phase 2 assignment: token e2 (+ 16 per pass), features f0 .. f0 + 7 and 64 + f0 .. 64 + f0 + 7
      const int e2 = st >> 3, f0 = (st & 7) * 8;
      const float* xlo = xset + (f0 >> 5) * QUARTER + (f0 & 31);
      const float* xhi = xset + (2 + (f0 >> 5)) * QUARTER + (f0 & 31);
      float* xmine = xset + quarter * QUARTER + lane;
      int it = 0;
      for (int u = pair; u < p.n_units; u += p.n_pairs, ++it) {
        const int b = it & 1;
        int fb, row0;
        sp_place<EPI>(p, u, fb, row0);
        const int hd = 2 * fb + (int)rank;
        const bool live = hd < p.n_heads;
        const int hde = live ? hd : 0;
        const int sg = (hde >= p.seg_heads_end[0]) + (hde >= p.seg_heads_end[1]);
        const int head_in_seg = hde - (sg == 0 ? 0 : p.seg_heads_end[sg - 1]);
        const int kind = p.kind[sg];
        const int t0 = row0 + set * set_n;
        const float bias = p.bias[sg] ? __bfloat162float(p.bias[sg][head_in_seg * 128 + quarter * 32 + lane]) : 0.f;
        const bool rotate = kind != 2;
        {  // positions of the set's tokens, checked: -1 where nothing is to be written
          int ps = -1;
          if (st < set_n && t0 + st < p.M) {
            ps = p.pos[t0 + st];
            if (ps < 0 || ps >= p.kv_len || ps >= p.max_pos) {
              if (live) atomicOr(p.status, A3_DEV_BAD_POSITION);
              ps = -1;
            }
          }
          posbuf[st] = live ? ps : -1;
        }
        named_bar_sync(bar_set, 128);
        // (cos, sin) of this thread's rotation pairs of a chunk: four vectors per pass.  Half-split pairs (i, i + 64): frequencies
        // f0 .. f0 + 7; adjacent pairs (2i, 2i + 1): f0/2 .. f0/2 + 3 for the first eight features, 32 higher for the others
        float4 tab[4 * PASSES];
        auto fetch = [&](int c) {
          if (!rotate) return;
#pragma unroll
          for (int pass = 0; pass < PASSES; ++pass) {
            const int e = c * CH + e2 + 16 * pass;
            const float2* row = p.tab + (size_t)max(posbuf[min(e, 127)], 0) * 64;
            const float4* lo = reinterpret_cast<const float4*>(row + (p.layout == 0 ? f0 : f0 >> 1));
            const float4* hi = reinterpret_cast<const float4*>(row + (p.layout == 0 ? f0 + 4 : 32 + (f0 >> 1)));
            ldg32(lo, tab[4 * pass], tab[4 * pass + 1]);
            ldg32(hi, tab[4 * pass + 2], tab[4 * pass + 3]);
          }
        };
        fetch(0);
        if (ep_tid == 0) ep_ok[0] = mbar_wait(tmem_full(b), (it >> 1) & 1, abort_flag, p.status) ? 1 : 0;
        named_bar_sync(1, 256);
        if (!ep_ok[0]) {  // uniform for the 256 threads
          give_up();
          return false;
        }
        tc_fence_after();
        const uint32_t trow = tmem_base + (uint32_t)(b * p.slot_cols) + (uint32_t)(set * set_n) + ((uint32_t)(quarter * 32) << 16);
        // KC > 1: [token of the set][128 features] fp32 sums of the other pair, over the ring, whose stages have all been read
        // once both pairs have published their accumulators
        const float* theirs = reinterpret_cast<const float*>(base_ptr) + quarter * 32 + lane;
        if constexpr (KC > 1) {
          __syncwarp();
          cluster_sync_all();
          if (set != kc) {
            uint32_t to;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(base + (uint32_t)(quarter * 32 + lane) * 4), "r"(crank ^ 2u));
#pragma unroll 1
            for (int c = 0; c < n_chunks; ++c) {
              float v[CH];
              __syncwarp();
              sp_ld_chunk<CH>(trow + c * CH, min(CH, set_n - c * CH), v);
#pragma unroll
              for (int e = 0; e < CH; ++e)
                if (c * CH + e < set_n)
                  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to + (uint32_t)(c * CH + e) * 512), "f"(v[e]) : "memory");
            }
          }
          __syncwarp();
          cluster_sync_all();
          merged = 2;
          if (set != kc) return true;
        }
#pragma unroll 1
        for (int c = 0; c < n_chunks; ++c) {
          float v[CH];
          __syncwarp();
          sp_ld_chunk<CH>(trow + c * CH, min(CH, set_n - c * CH), v);
          if constexpr (KC > 1) {
#pragma unroll
            for (int e = 0; e < CH; ++e)
              if (c * CH + e < set_n) v[e] += theirs[(c * CH + e) * 128];
          }
#pragma unroll
          for (int e = 0; e < CH; ++e) xmine[e * 32] = v[e] + bias;
          named_bar_sync(bar_set, 128);
          uint4 out_lo[PASSES], out_hi[PASSES];
#pragma unroll
          for (int pass = 0; pass < PASSES; ++pass) {
            const int e = e2 + 16 * pass;
            float a[8], bq[8], ra[8], rb[8];
            *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(xlo + e * 32);
            *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(xlo + e * 32 + 4);
            *reinterpret_cast<float4*>(bq) = *reinterpret_cast<const float4*>(xhi + e * 32);
            *reinterpret_cast<float4*>(bq + 4) = *reinterpret_cast<const float4*>(xhi + e * 32 + 4);
            if (!rotate) {
#pragma unroll
              for (int k = 0; k < 8; ++k) ra[k] = a[k], rb[k] = bq[k];
            } else if (p.layout == 0) {
              // the thread's first 8 features rotate with the 8 that lie 64 further
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const float4 t = tab[4 * pass + k];  // (cos, sin) of two frequencies
                ra[2 * k] = a[2 * k] * t.x - bq[2 * k] * t.y;
                rb[2 * k] = a[2 * k] * t.y + bq[2 * k] * t.x;
                ra[2 * k + 1] = a[2 * k + 1] * t.z - bq[2 * k + 1] * t.w;
                rb[2 * k + 1] = a[2 * k + 1] * t.w + bq[2 * k + 1] * t.z;
              }
            } else {
              // both groups of 8 hold four pairs of their own
#pragma unroll
              for (int k = 0; k < 2; ++k) {
                const float4 t = tab[4 * pass + k], u4 = tab[4 * pass + 2 + k];
                ra[4 * k] = a[4 * k] * t.x - a[4 * k + 1] * t.y;
                ra[4 * k + 1] = a[4 * k] * t.y + a[4 * k + 1] * t.x;
                ra[4 * k + 2] = a[4 * k + 2] * t.z - a[4 * k + 3] * t.w;
                ra[4 * k + 3] = a[4 * k + 2] * t.w + a[4 * k + 3] * t.z;
                rb[4 * k] = bq[4 * k] * u4.x - bq[4 * k + 1] * u4.y;
                rb[4 * k + 1] = bq[4 * k] * u4.y + bq[4 * k + 1] * u4.x;
                rb[4 * k + 2] = bq[4 * k + 2] * u4.z - bq[4 * k + 3] * u4.w;
                rb[4 * k + 3] = bq[4 * k + 2] * u4.w + bq[4 * k + 3] * u4.z;
              }
            }
            out_lo[pass] = pack8(ra);
            out_hi[pass] = pack8(rb);
          }
          if (c + 1 < n_chunks) fetch(c + 1);
#pragma unroll
          for (int pass = 0; pass < PASSES; ++pass) {
            const int e = c * CH + e2 + 16 * pass;
            const int ps = e < set_n ? posbuf[e] : -1;
            if (ps < 0) continue;
            bf16* dst = kind == 0 ? p.q_out + (size_t)(t0 + e - p.q_first) * (p.Hq * 128) + head_in_seg * 128
                      : (kind == 1 ? p.k_cache : p.v_cache) + (size_t)ps * (p.Hkv * 128) + head_in_seg * 128;
            *reinterpret_cast<uint4*>(dst + f0) = out_lo[pass];
            *reinterpret_cast<uint4*>(dst + 64 + f0) = out_hi[pass];
          }
          named_bar_sync(bar_set, 128);  // everybody has read this chunk's values and positions
        }
        // this warp has read its part of the accumulator (wait::ld in sp_ld_chunk): it goes back to the MMA issuer
        tc_fence_before();
        __syncwarp();
        if (lane == 0 && awaited(it)) mbar_arrive_in_cta(tmem_empty(b), pair_cta0);
      }
      return true;
    });
  } else if (EPI == EPI_RESIDUAL) {
    // ---------------- epilogue, C += A B^T: warps 2..9 of both CTAs; warp w may touch TMEM lanes 32*(w%4) .. +31,
    // lane = output feature; warp set 0 (warps 2..5) takes the first half of the token columns, set 1 the second.  A chunk of
    // tokens at a time in the two phases of the QKV epilogue: feature-major out of tensor memory into shared memory, then
    // token-major, a thread taking 8 consecutive features of a token (16 bytes of C, 256 contiguous bytes per token).
    // All old values of a unit (at most 16 vectors per thread) are requested while its main loop still runs: a launch with
    // one unit per pair has nothing else to hide them under.
    const int quarter = warp & 3;
    const int set = (warp - 2) >> 2;
    const int ep_tid = (warp - 2) * 32 + lane;
    const int st = quarter * 32 + lane;  // thread within the set
    const int set_n = p.tok_n >> 1;
    const int bar_set = 2 + set;
    // phase 2 assignment: tokens e2, e2 + 8, .. of a chunk, features 8 (st & 15) .. + 7
    const int e2 = st >> 4, fg = st & 15;
    sp_with_chunk<true>(p.chunk, [&](auto chunk) {
      constexpr int CH = decltype(chunk)::value, QUARTER = CH * 32 + 4;
      const int n_chunks = (set_n + CH - 1) / CH;
      float* xset = xch + set * sp_set_floats(CH);
      float* xmine = xset + quarter * QUARTER + lane;
      const float* xrow = xset + (fg >> 2) * QUARTER + (fg & 3) * 8;
      int it = 0;
      for (int u = pair; u < p.n_units; u += p.n_pairs, ++it) {
        const int b = it & 1;
        int fb, tt;
        sp_unit(u, p.n_fblocks, p.tok_tiles, p.group, fb, tt);
        const int f = fb * (2 * ROWS) + (int)rank * ROWS + fg * 8;
        const int t0 = tt * p.tok_n + set * set_n;
        // tokens of this set that exist; none where the last feature block reaches past the matrix (zero-filled loads)
        const int valid = f < p.F ? min(set_n, p.M - t0) : 0;
        bf16* crow = p.C + (size_t)(valid > 0 ? t0 : 0) * p.ldc + (valid > 0 ? f : 0);
        uint4 old[16];
#pragma unroll
        for (int i = 0; i < 16; ++i)
          old[i] = i * 8 + e2 < valid ? __ldcg(reinterpret_cast<const uint4*>(crow + (size_t)(i * 8 + e2) * p.ldc)) : make_uint4(0, 0, 0, 0);
        if (ep_tid == 0) ep_ok[0] = mbar_wait(tmem_full(b), (it >> 1) & 1, abort_flag, p.status) ? 1 : 0;
        named_bar_sync(1, 256);
        if (!ep_ok[0]) {  // uniform for the 256 threads
          give_up();
          return false;
        }
        tc_fence_after();
        const uint32_t trow = tmem_base + (uint32_t)(b * p.slot_cols) + (uint32_t)(set * set_n) + ((uint32_t)(quarter * 32) << 16);
#pragma unroll
        for (int c = 0; c < 128 / CH; ++c) {
          if (c >= n_chunks) break;
          float v[CH];
          __syncwarp();
          sp_ld_chunk<CH>(trow + c * CH, min(CH, set_n - c * CH), v);
#pragma unroll
          for (int e = 0; e < CH; ++e) xmine[e * 32] = v[e];
          named_bar_sync(bar_set, 128);
#pragma unroll
          for (int i = 0; i < CH / 8; ++i) {
            const int e = i * 8 + e2;
            if (c * CH + e >= valid) continue;
            float a[8], o[8];
            *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(xrow + e * 32);
            *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(xrow + e * 32 + 4);
            unpack8(old[c * (CH / 8) + i], o);
#pragma unroll
            for (int k = 0; k < 8; ++k) a[k] += o[k];
            *reinterpret_cast<uint4*>(crow + (size_t)(c * CH + e) * p.ldc) = pack8(a);
          }
          named_bar_sync(bar_set, 128);  // everybody has read this chunk's values
        }
        // this warp has read its part of the accumulator (wait::ld in sp_ld_chunk): it goes back to the MMA issuer
        tc_fence_before();
        __syncwarp();
        if (lane == 0 && awaited(it)) mbar_arrive_in_cta(tmem_empty(b), pair_cta0);
      }
      return true;
    });
  }
  if constexpr (KC > 1) {  // the warps without a part in the merge, and everybody after a wait that gave up
    __syncwarp();
    for (; merged < 2; ++merged) cluster_sync_all();
  }
  tc_fence_before();
  // Neither CTA releases tensor or shared memory while the other may still use it.  Ordering execution is enough: the stores above
  // are for the kernels that follow, and a barrier that releases them first waited 700-900 clocks for their way to L2 in
  // every launch.  Request of 369 tokens on a small model 153.2 -> 146.1 us, prefill of 75 tokens (Qwen-7B) 2 924 -> 2 873, request
  // of three passages (Llama-8B) 4 277 -> 4 219.  Arrivals at the leader that it does not wait for are ordered where they are given up.
  cluster_sync_relaxed();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
}

// A3_OPT_SWIGLU_PAIR / A3_OPT_RESIDUAL_T: 0 never; 1 whenever the shape allows (default); cross-checks switch them off
// to compare with the other kernels
bool swiglu_pair_usable(const a3_handle* h, const GemmArgs& a) {
  return h->opt[A3_OPT_SWIGLU_PAIR] != 0 && a.M > 0 && a.K % (SP_SUB * TC_BK) == 0 && a.seg[0].n % (2 * SP_FEAT) == 0 && a.seg[0].bias == nullptr;
}
// A3_OPT_RESIDUAL_T: 0 never, otherwise whenever the shape allows.  Against the 256 x 256 tile kernel, output + down projection
// of a layer: 513 rows 110 -> 81 us, 804 rows 116 -> 105, 1 024 rows 118 -> 119 (Llama width); 550 rows 133 -> 94, 804 rows
// 142 -> 110 (Qwen width).
bool residual_t_usable(const a3_handle* h, const GemmArgs& a) {
  return h->opt[A3_OPT_RESIDUAL_T] != 0 && a.M > 0 && a.K % (SP_SUB * TC_BK) == 0 && a.nseg == 1 && a.seg[0].n % 32 == 0 &&
         a.seg[0].bias == nullptr;
}

// Token tiling of a launch: `tiles` tiles of `n` tokens (a multiple of 16, at most 256) that divide the row count
// evenly.  The tile count is the one with the cheapest rounds: the CTA pairs take the units (feature block x token
// tile) round by round, and a unit of n token columns costs, per k-block, the larger of its tensor time (2 n clocks:
// four instructions of n / 2) and the time its operands take to arrive (16 KiB of weights + 64 n bytes of tokens per
// CTA at about 64 bytes per clock: 256 + n clocks), plus a fixed part.  By that measure every unit narrower than 256
// waits for its operands, and the measurements agree: 804 rows x 112 feature blocks as five tiles of 176 (or as
// 4 x 176 + 112 with the narrow units last, which a count of token columns alone prefers) took 160-165 us against 147
// for 4 x 208.  Examples: 4 952 rows x 16 feature blocks -> 23 x 224 (five rounds of 224 instead of five of 256:
// 536 vs 591 us for both residual GEMMs of a layer), x 112 -> 20 x 256 as before; 804 rows x 24 head pairs -> 6 x 144
// (two rounds) instead of 4 x 208 (two rounds).  A3_OPT_GEMM_TILING = 1 keeps ceil(M / 256) tiles (comparisons).
// Feature blocks per group of the unit order: 8 when the token matrix (M x K bf16) is too large to stay in L2 beside
// the weights and the output that stream through it, else 1.
static int unit_group(int M, int K) { return (long long)M * K * 2 > (64ll << 20) ? 8 : 1; }

// Two token tiles of n per unit on one stream of weights.  Just over 256 rows every weight goes to two units, and units that narrow
// wait for their operands: 270 rows x 2 x (16 KiB of weights + 9 KiB of tokens) per k-block and CTA, 800 clocks for 576 of tensor time.
// Together they take 16 + 18 KiB, 576 clocks of tensor time, and each weight crosses to an SM once: inside a request of 270 rows (Qwen
// width) SwiGLU 67 -> 57 us, down projection 42 -> 31.5; SwiGLU alone 65.4 -> 62.7.
constexpr int SP_TWO_TILES_COLS = 160;  // columns from one accumulator to the next: three in 512
constexpr int SP_TWO_TILES_MAX = 144;   // tokens per tile of SwiGLU, see two_tiles
static int two_tiles_per_kb(int n) { return 4 * n > 256 + 2 * n ? 4 * n : 256 + 2 * n; }

struct SpTiling {
  int tiles, n;
};
static SpTiling choose_tiling(const a3_handle* h, int M, int n_fblocks, int pairs) {
  SpTiling best{cdiv(M, 256), 0};
  best.n = cdiv(cdiv(M, best.tiles), 16) * 16;  // 804 rows -> 4 x 208
  if (h->opt[A3_OPT_GEMM_TILING] == 1) return best;
  auto load = [&](int tiles, int n) {
    const long long unit = (long long)(2 * n > 256 + n ? 2 * n : 256 + n) + 32;
    return (long long)cdiv((long long)n_fblocks * tiles, pairs) * unit;
  };
  long long best_load = load(best.tiles, best.n);
  for (int tiles = best.tiles + 1; tiles <= best.tiles + 64 && tiles <= cdiv(M, 96); ++tiles) {
    const int n = cdiv(cdiv(M, tiles), 16) * 16;
    const long long l = load(tiles, n);
    if (l < best_load) {
      best_load = l;
      best = SpTiling{tiles, n};
    }
  }
  return best;
}

// How many k-slices the residual GEMM of few rows is cut into (1: not at all).  With one unit per 256 features x 256
// tokens, M <= 512 rows leave most of the 74 CTA pairs idle: a down projection of 75 rows x 3 584 features ran on 28 SMs
// and streamed its 136 MB of weights at 1.4 TB/s.  Compared are, in clocks, one round of whole units and rounds of the
// split ones (a k-block costs the larger of its tensor time and the arrival of its operands, see choose_tiling) plus the
// fp32 partial sums, which are written and read once each through L2 (about 3 KB a clock), at most `part_bytes` of them.
// A slice is at least 1 024 deep: shorter ones are all pipeline fill.
// Pinned kernel variants (a3_set_option) are compared bit for bit and therefore keep the undivided sums.
constexpr int SP_SLICE_MIN_KB = 16;
static bool split_allowed(const a3_handle* h) {
  return (h->opt[A3_OPT_RESIDUAL_T] == 1 || h->opt[A3_OPT_RESIDUAL_T] == 3) && h->opt[A3_OPT_QKV_T] == 1 && h->opt[A3_OPT_SWIGLU_PAIR] == 1 &&
         h->opt[A3_OPT_GEMM_TILING] == 0;
}
struct SpSlices {
  int slices, tiles;  // tiles: token tiles per unit
};
static SpSlices choose_slices(int M, int F, int K, int n_fblocks, int pairs, size_t part_bytes) {
  const int tiles = cdiv(M, 256), n = cdiv(cdiv(M, tiles), 16) * 16, kt = K / TC_BK;
  const int per_kb = 2 * n > 256 + n ? 2 * n : 256 + n;
  auto depth = [&](int s) { return (long long)cdiv(kt / SP_SUB, s) * SP_SUB; };  // k-blocks of the deepest slice
  auto sums = [&](int s) { return (long long)s * M * F * 8 / 3000 + 2000; };
  long long least = (long long)kt * per_kb;
  SpSlices best{1, 1};
  for (int s = 2; s <= 16 && s * SP_SLICE_MIN_KB <= kt; ++s) {
    if ((size_t)s * M * F * 4 > part_bytes) break;
    const long long cost = (long long)cdiv((long long)n_fblocks * tiles * s, pairs) * (depth(s) * per_kb + 2000) + sums(s);
    if (cost < least) {
      least = cost;
      best = SpSlices{s, 1};
    }
  }
  // The same slices with both tiles on one stream of weights (two_tiles), one unit per pair: both accumulators of 256 columns are in
  // use.  Not with more slices for the sake of it, which would change the sums and lost where it was tried: a layer of 257 rows in two
  // slices against five of two tiles 103.7 / 105.1 us at 3 200 x 10 112, 106.9 / 107.6 at 3 328 x 10 624; prefill (us) of Llama-8B in
  // two slices against four, 272 rows 5 200 / 5 231, 320 rows 5 486 / 5 547.  Qwen-7B, five slices either way: a layer 156.4 / 150.9
  // at 257 rows, 163.9 / 158.8 at 272, 175.6 / 172.1 at 320, 192.9 / 191.7 at 352, hence the tenth that is left out.
  if (tiles == 2 && best.slices > 1 && n_fblocks * best.slices <= pairs &&
      (depth(best.slices) * two_tiles_per_kb(n) + 2000 + n * 20 + sums(best.slices)) * 10 < least * 9)
    best.tiles = 2;
  return best;
}
int residual_slices(const a3_handle* h, int M, int N, int K, size_t part_bytes, int* tiles) {
  *tiles = 1;
  if (!split_allowed(h) || h->opt[A3_OPT_GEMM_BN_RESIDUAL] != 0 || M <= 0 || K % (SP_SUB * TC_BK) || N % 32) return 1;
  const int pairs = (h->sm_count > 0 ? h->sm_count : 148) / 2, blocks = cdiv(N, 4 * SP_FEAT);
  if (blocks * cdiv(M, 256) > pairs / 2) return 1;  // the pairs are busy with whole units
  const SpSlices c = choose_slices(M, N, K, blocks, pairs, part_bytes);
  *tiles = h->opt[A3_OPT_RESIDUAL_T] == 3 ? 1 : c.tiles;
  return c.slices;
}

// Weights that nobody finds in L2 again: one token tile, so that the launch reads each of them once, and a stack of layers
// beyond L2, so that the next request does not either.  A model that L2 holds wants its weights left there.  One layer back to
// back, normal policy against marked weights (us, 13 / 75 / 200 rows): 78 MB 40.7 / 47.0 / 65.0 against 44.8 / 51.0 / 64.8; 90 MB
// 42.7 / 49.7 / 69.4 and 46.9 / 53.5 / 71.4; 100 MB 44.8 / 52.0 / 73.2 and 48.9 / 55.5 / 71.4; 115 MB 50.9 / 58.9 / 76.0 and
// 51.0 / 57.1 / 73.5; 131 MB 55.5 / 61.9 / 78.0 and 53.0 / 59.6 / 74.0; with heads of 64, 122 MB 66.1 / 72.0 / 85.5 and
// 59.1 / 64.2 / 75.5; 18 MB in three layers no difference.  Hence the line at three quarters of L2.  The QKV projection in
// clusters marks its weights always: with the normal policy the 90 MB layer took 43.3 and 50.4 us for 13 and 75 rows.
static bool weights_once(const a3_handle* h, int tok_tiles) { return tok_tiles == 1 && h->stack_over_l2; }

// Ring depth and epilogue chunk of a launch: the widest chunk among those that leave the ring deepest (a stage more is 8 %
// at 513 rows, where 32-token chunks leave three stages of 176 tokens and 8-token chunks four), but no deeper than a pair
// has stages to run through.  Returns the dynamic shared memory.
static int set_stages(SpParams& p, int epi, bool split, int tt = 1) {
  const int sub = SP_SUB / tt;
  p.stage_bytes = sub * (SP_A_BYTES + tt * (p.tok_n / 2) * TC_BK * 2);  // tok_n / 2 is a multiple of 8: 1024-byte multiples
  p.slot_cols = tt == 1 || split ? 256 : SP_TWO_TILES_COLS;
  p.stages = 0;
  const long long steps = (long long)cdiv(p.n_units, p.n_pairs) * (p.K / TC_BK / sub);
  const int useful = steps < SP_MAX_STAGES ? (int)steps : SP_MAX_STAGES;
  int xch = 0;
  for (int chunk = 32; chunk >= (epi == EPI_QKV || tt == 2 ? 16 : 8); chunk /= 2) {
    const int x = split ? 0 : sp_xch_bytes(epi, chunk);
    int stages = (SP_SMEM_LIMIT - x - 256) / p.stage_bytes;
    if (stages > useful) stages = useful;
    if (stages > p.stages) {
      p.stages = stages;
      p.chunk = chunk;
      xch = x;
    }
  }
  return p.stages * p.stage_bytes + xch + 256;
}

int gemm_residual_split(const a3_handle* h, const GemmArgs& a, int slices, int tiles, float* part, cudaStream_t st) {
  SpParams p{};
  p.M = a.M;
  p.K = a.K;
  p.F = a.seg[0].n;
  const int pairs = (h->sm_count > 0 ? h->sm_count : 148) / 2;
  p.n_fblocks = cdiv(p.F, 4 * SP_FEAT);
  p.tok_tiles = cdiv(a.M, 256);
  p.tok_n = cdiv(cdiv(a.M, p.tok_tiles), 16) * 16;
  if (tiles == 2) p.tok_tiles = 1;
  p.k_slices = slices;
  p.early = a.early_weights;
  p.part = part;
  p.n_units = p.n_fblocks * p.tok_tiles * slices;
  p.group = 1;
  // two tiles: accumulators of 256 columns, of which tensor memory holds two, so one unit per pair (choose_slices sees to both)
  if (tiles == 2 && (p.n_units > pairs || a.M <= 256 || a.M > 512)) return A3_EINVAL;
  p.n_pairs = p.n_units < pairs ? p.n_units : pairs;
  p.status = h->dev_status;
  const int smem_bytes = set_stages(p, EPI_RESIDUAL, true, tiles);
  CUtensorMap tX, tG;
  A3_TRY(make_tmap_kblocks(&tX, a.A, a.M, a.K, p.tok_n / 2, SP_SUB / tiles));
  A3_TRY(make_tmap_kblocks(&tG, a.seg[0].B, p.F, a.K, 2 * SP_FEAT, SP_SUB / tiles));
  // (Two tiles mark their weights always: the smallest layer that takes them is more than twice L2.)
  static SmemAttrOnce attr[3];
  const int variant = tiles == 2 ? 2 : weights_once(h, p.tok_tiles);
  const auto kernel = variant == 2   ? pair_t_kernel<EPI_RESIDUAL, true, 1, true, 2>
                      : variant == 1 ? pair_t_kernel<EPI_RESIDUAL, true, 1, true>
                                     : pair_t_kernel<EPI_RESIDUAL, true, 1, false>;
  A3_TRY(smem_attr_once(attr[variant], h->device, kernel, SP_SMEM_LIMIT));
  ProfScope prof(h, A3_K_GEMM_RESIDUAL, st);
  A3_CUDA(launch_pdl(kernel, dim3(2 * p.n_pairs), dim3(SP_THREADS), (size_t)smem_bytes, st, tX, tG, tG, tG, p));
  A3_LAUNCHED();
  return A3_OK;
}

// SwiGLU on two token tiles per unit: every unit costs half an epilogue more, which the third accumulator does not hide, and a k-block
// a fifth more than its operands take to arrive.  One layer of a stack beyond L2, one tile per unit against two (us): Llama-8B 257 rows
// 142.1 / 137.6, 272 155.7 / 154.7, 288 157.3 / 156.1; Qwen-7B 257 rows 153.3 / 150.9, 272 159.8 / 158.8; 3 072 x 8 192 257 rows 85.3 /
// 83.8, 288 88.1 / 87.0.  Where the model says one: 2 048 x 16 384 257 rows 92.9 / 94.5, 2 048 x 8 192 71.9 / 71.5 (SwiGLU alone, from
// L2, 16.6 / 19.2), 1 536 x 8 960 62.0 / 61.3 (13.8 / 15.6).  Tiles of 160 lost at every width but the narrowest: 304 and 320 rows,
// Llama-8B 163.7 / 167.2 and 162.3 / 166.4, Qwen-7B 163.6 / 165.3 and 169.1 / 172.1, 2 048 x 16 384 94.3 / 96.9 and 97.2 / 101.2.  The
// epilogue's chunks stay at 16 tokens or more: with 8, for the sake of one ring stage more, nothing was gained.
static bool two_tiles(const a3_handle* h, int M, int K, int n_fblocks, int pairs, const SpTiling& til) {
  const int n = cdiv(cdiv(M, 2), 16) * 16, kt = K / TC_BK;
  if (M <= 256 || n > SP_TWO_TILES_MAX || h->opt[A3_OPT_GEMM_TILING] != 0) return false;
  const int per_kb = 2 * til.n > 256 + til.n ? 2 * til.n : 256 + til.n;
  return (long long)cdiv(n_fblocks, pairs) * (kt * two_tiles_per_kb(n) * 6 / 5 + 30 * n) < (long long)cdiv((long long)n_fblocks * til.tiles, pairs) * kt * per_kb;
}

// Token tiles per unit of the gate/up GEMM by default (a3_plan_layer)
int swiglu_tiles(const a3_handle* h, int M, int K, int F) {
  const int pairs = (h->sm_count > 0 ? h->sm_count : 148) / 2, n_fblocks = cdiv(F, 2 * SP_FEAT);
  return M > 0 && two_tiles(h, M, K, n_fblocks, pairs, choose_tiling(h, M, n_fblocks, pairs)) ? 2 : 1;
}

template <int EPI>
static int launch_pair_t(const a3_handle* h, const GemmArgs& a, cudaStream_t st) {
  constexpr int ROWS = EPI == EPI_SWIGLU ? SP_FEAT : 2 * SP_FEAT;  // output features per CTA
  SpParams p{};
  p.M = a.M;
  p.K = a.K;
  p.F = a.seg[0].n;
  const int sms = h->sm_count > 0 ? h->sm_count : 148;
  p.n_fblocks = cdiv(p.F, 2 * ROWS);
  const SpTiling til = choose_tiling(h, a.M, p.n_fblocks, sms / 2);
  const int tt = EPI == EPI_SWIGLU && two_tiles(h, a.M, a.K, p.n_fblocks, sms / 2, til) ? 2 : 1;
  p.tok_tiles = tt == 2 ? 1 : til.tiles;
  p.tok_n = tt == 2 ? cdiv(cdiv(a.M, 2), 16) * 16 : til.n;
  p.n_units = p.n_fblocks * p.tok_tiles;
  p.group = unit_group(a.M, a.K);
  p.k_slices = 1;
  p.early = a.early_weights;
  p.n_pairs = p.n_units < sms / 2 ? p.n_units : sms / 2;
  p.C = a.C;
  p.ldc = a.ldc;
  p.status = h->dev_status;
  const int smem_bytes = set_stages(p, EPI, false, tt);
  CUtensorMap tX, tG, tU;
  A3_TRY(make_tmap_kblocks(&tX, a.A, a.M, a.K, p.tok_n / 2, SP_SUB / tt));
  A3_TRY(make_tmap_kblocks(&tG, a.seg[0].B, p.F, a.K, ROWS, EPI == EPI_SWIGLU ? 1 : SP_SUB));
  if (EPI == EPI_SWIGLU) A3_TRY(make_tmap_kblocks(&tU, a.B2, p.F, a.K, ROWS, 1));
  else tU = tG;
  static SmemAttrOnce attr[4];
  const bool once = weights_once(h, p.tok_tiles);
  auto kernel = once ? pair_t_kernel<EPI, false, 1, true> : pair_t_kernel<EPI, false, 1, false>;
  if constexpr (EPI == EPI_SWIGLU) {
    if (tt == 2) kernel = once ? pair_t_kernel<EPI, false, 1, true, 2> : pair_t_kernel<EPI, false, 1, false, 2>;
  }
  A3_TRY(smem_attr_once(attr[2 * (tt - 1) + once], h->device, kernel, SP_SMEM_LIMIT));
  ProfScope prof(h, EPI == EPI_SWIGLU ? A3_K_GEMM_SWIGLU : A3_K_GEMM_RESIDUAL, st);
  A3_CUDA(launch_pdl(kernel, dim3(2 * p.n_pairs), dim3(SP_THREADS), (size_t)smem_bytes, st, tX, tG, tU, tU, p));
  A3_LAUNCHED();
  return A3_OK;
}

// QKV projection on the same kernel: one head (128 features) per CTA of a pair, token tiles chosen so that the units
// fill whole rounds of the CTA pairs.  A3_OPT_QKV_T: 0 never, 1 whenever the shape allows (default).
bool qkv_t_usable(const a3_handle* h, const GemmArgs& a) {
  if (h->opt[A3_OPT_QKV_T] == 0 || h->m.head_dim != 128 || a.M <= 0 || a.K % (SP_SUB * TC_BK) != 0 || a.nseg < 1 || a.nseg > 3) return false;
  for (int s = 0; s < a.nseg; ++s)
    if (a.seg[s].n % 128 != 0 || a.seg[s].n <= 0) return false;
  if (a.q_first > 0) {
    // Late queries ride along where the K/V units leave room in their last round (a round more costs what a launch of its own
    // does, or more: its units are as wide as the K/V tiles).  A request
    // of 369 tokens on a small model 159.5 -> 157.0 us.
    if (a.nseg != 3 || a.seg[0].kind != 1 || a.seg[1].kind != 2 || a.seg[2].kind != 0 || a.q_first >= a.M) return false;
    if ((a.seg[0].n + a.seg[1].n) % 256 != 0) return false;
    const int pairs = (h->sm_count > 0 ? h->sm_count : 148) / 2, kv_pairs = (a.seg[0].n + a.seg[1].n) / 256;
    const SpTiling til = choose_tiling(h, a.M, kv_pairs, pairs);
    const int kv_units = kv_pairs * til.tiles, q_units = cdiv(a.seg[2].n, 256) * cdiv(a.M - a.q_first, til.n);
    return cdiv(kv_units + q_units, pairs) == cdiv(kv_units, pairs);
  }
  return true;
}

// QKV of few rows in clusters of two pairs, each with half of the k-loop.  The heads alone occupy few pairs (Llama-8B: 24,
// Qwen-7B: 18 of 74) and a CTA takes in its 16 KiB of weights per k-block at about 107 GB/s, however fast HBM is: 9.5 us for
// the 33 MB of Qwen-7B.  Halves stream twice as wide; the merge costs two cluster barriers and a trip of the sums through
// distributed shared memory (about 2 500 clocks).  Compared with the other way to occupy pairs, narrower token tiles, by the
// cost per k-block of choose_tiling.  A layer of 75 rows (Qwen width) 88.8 -> 87.5 us, of 144 rows (Llama width) 111.6 ->
// 109.6.  A half is at least as deep as a slice of the residual GEMMs; a tenth of the pairs is left out because clusters of
// four do not fill every GPC.  Pinned kernel variants keep the undivided sums (split_allowed).
static bool qkv_clusters(const a3_handle* h, int M, int K, int head_pairs, int pairs, const SpTiling& til) {
  if (!split_allowed(h) || M > 256 || 2 * head_pairs > pairs - pairs / 10 || K / TC_BK < 2 * SP_SLICE_MIN_KB) return false;
  auto per_kb = [](int n) { return 2 * n > 256 + n ? 2 * n : 256 + n; };
  const int kt = K / TC_BK;
  return kt / 2 * per_kb(cdiv(M, 16) * 16) + 2500 < (long long)cdiv(head_pairs * til.tiles, pairs) * kt * per_kb(til.n);
}

int gemm_qkv_t(const a3_handle* h, const GemmArgs& a, cudaStream_t st) {
  SpParams p{};
  p.M = a.M;
  p.K = a.K;
  int heads = 0;
  for (int s = 0; s < 3; ++s) {
    if (s < a.nseg) {
      heads += a.seg[s].n / 128;
      p.kind[s] = a.seg[s].kind;
      p.bias[s] = a.seg[s].bias;
    }
    p.seg_heads_end[s] = heads;
  }
  p.n_heads = heads;
  const int kv_heads = a.seg[0].n / 128 + (a.nseg > 1 ? a.seg[1].n / 128 : 0);
  const int head_pairs = a.q_first > 0 ? kv_heads / 2 : cdiv(heads, 2);  // of the units over all rows
  const int sms = h->sm_count > 0 ? h->sm_count : 148;
  const int pairs = sms / 2;
  const SpTiling til = choose_tiling(h, a.M, head_pairs, pairs);
  const bool clusters = a.q_first == 0 && qkv_clusters(h, a.M, a.K, head_pairs, pairs, til);
  p.tok_tiles = clusters ? 1 : til.tiles;
  p.tok_n = clusters ? cdiv(a.M, 16) * 16 : til.n;
  p.n_fblocks = head_pairs;
  p.group = unit_group(a.M, a.K);
  p.k_slices = 1;
  p.early = a.early_weights;
  p.n_units = p.q_unit0 = head_pairs * p.tok_tiles;
  p.q_first = a.q_first;
  if (a.q_first > 0) {
    p.q_block0 = head_pairs;
    p.q_tiles = cdiv(a.M - a.q_first, p.tok_n);
    p.n_units += cdiv(a.seg[2].n / 128, 2) * p.q_tiles;
  }
  p.n_pairs = p.n_units < pairs ? p.n_units : pairs;
  p.status = h->dev_status;
  p.q_out = a.q_out;
  p.k_cache = a.k_cache;
  p.v_cache = a.v_cache;
  p.pos = a.pos;
  p.kv_len = a.kv_len;
  p.Hq = h->m.n_q_heads;
  p.Hkv = h->m.n_kv_heads;
  p.layout = h->m.rope_layout;
  p.max_pos = h->m.max_positions;
  p.tab = h->rope_tab;
  const int smem_bytes = set_stages(p, EPI_QKV, false);
  CUtensorMap tX, tW[3];
  A3_TRY(make_tmap_kblocks(&tX, a.A, a.M, a.K, p.tok_n / 2, SP_SUB));
  for (int s = 0; s < 3; ++s) {
    if (s < a.nseg) A3_TRY(make_tmap_kblocks(&tW[s], a.seg[s].B, a.seg[s].n, a.K, 128, SP_SUB));
    else tW[s] = tW[0];
  }
  static SmemAttrOnce attr[3];
  const int variant = clusters ? 2 : weights_once(h, p.tok_tiles);
  const auto kernel = variant == 2   ? pair_t_kernel<EPI_QKV, false, 2, true>
                      : variant == 1 ? pair_t_kernel<EPI_QKV, false, 1, true>
                                     : pair_t_kernel<EPI_QKV, false, 1, false>;
  A3_TRY(smem_attr_once(attr[variant], h->device, kernel, SP_SMEM_LIMIT));
  ProfScope prof(h, A3_K_GEMM_QKV, st);
  A3_CUDA(launch_pdl(kernel, dim3((clusters ? 4 : 2) * p.n_pairs), dim3(SP_THREADS), (size_t)smem_bytes, st, tX, tW[0], tW[1], tW[2], p));
  A3_LAUNCHED();
  return A3_OK;
}

int gemm_swiglu_pair(const a3_handle* h, const GemmArgs& a, cudaStream_t st) { return launch_pair_t<EPI_SWIGLU>(h, a, st); }
int gemm_residual_t(const a3_handle* h, const GemmArgs& a, cudaStream_t st) { return launch_pair_t<EPI_RESIDUAL>(h, a, st); }

}  // namespace a3

// The gate/up GEMM of one layer alone (a3_swiglu_rows): out[M][d_ff] = silu(x Wg^T) * (x Wu^T), x [M][d_model].
extern "C" int a3_swiglu_rows(const a3_handle* h, int layer, const void* x, void* out, int M, a3_stream stream) {
  if (!h || layer < 0 || layer >= h->m.n_layers || M < 0) return A3_EINVAL;
  if (M == 0) return A3_OK;
  if (!x || !out || (((uintptr_t)x | (uintptr_t)out) & 15)) return A3_EINVAL;
  a3::GemmArgs u{};
  u.A = (const bf16*)x;
  u.M = M;
  u.K = h->m.d_model;
  u.nseg = 1;
  u.seg[0] = {(const bf16*)h->layers[layer].w_gate, nullptr, h->m.d_ff, 0};
  u.B2 = (const bf16*)h->layers[layer].w_up;
  u.C = (bf16*)out;
  u.ldc = h->m.d_ff;
  return a3::gemm_bf16(h, a3::EPI_SWIGLU, u, (cudaStream_t)stream);
}
