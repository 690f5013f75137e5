// Selection Re = top_p(s) (Eq. 3): block-radix select on the order-preserving integer image of the fp32 scores.
// One CTA per score array.  The scores are read from global memory once, as integer keys into registers (up to 8 192, see
// topk_regs) or shared memory (up to TK_SMEM_KEYS of them; longer arrays are re-read from global memory in every pass).  Up to four 8-bit histogram passes
// find the key of the k-th largest score: the warps count into TK_HISTS private histograms (a warp whose lanes all
// hold the same digit - the rule in the first pass, since the scores of one request share their leading bits - adds
// 32 with one instruction instead of serialising 32 atomics on one bin), the histograms are summed, and the bin of
// the k-th element is found by a parallel suffix sum over the 256 bins.  The emission is
// ordered: every warp (in registers: every thread) owns a contiguous span of the slots, counts what it will emit, and after one exchange of the
// 32 warp totals writes every slot above the threshold key plus, in slot order, as many slots equal to it as are
// still needed.  The result is exact: ties go to the lower slot and the output is ascending.
#include "a3_internal.cuh"

namespace a3 {

constexpr int TK_THREADS = 1024;
constexpr int TK_WARPS = TK_THREADS / 32;
constexpr int TK_HISTS = 16;              // private histograms (warp w counts into number w % TK_HISTS)
constexpr int TK_SMEM_KEYS = 48 * 1024;  // 192 KiB of keys

__device__ __forceinline__ uint32_t score_key(float s) {
  uint32_t u = __float_as_uint(s);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);  // larger float <=> larger key
}

// Sums the private histograms and finds the bin of the element of rank `remaining` (1-based, from the top); the caller's
// prefix, remaining and count (of the keys in the bin) move on to that bin.  All threads.
__device__ __forceinline__ void topk_bin(unsigned int (*whist)[256], unsigned int* warp_tot, unsigned int* s_prefix, unsigned int* s_remaining,
                                         unsigned int* s_count, int shift, uint32_t& prefix, unsigned int& remaining, unsigned int& count) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned int v = 0;
  if (tid < 256) {
#pragma unroll
    for (int w = 0; w < TK_HISTS; ++w) v += whist[w][tid];
    // suffix sums over the bins: S[d] = count of elements with digit >= d; the k-th element's digit is the largest d
    // with S[d] >= remaining
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int t = __shfl_down_sync(0xffffffffu, v, o);
      if (lane + o < 32) v += t;
    }
    if (lane == 0) warp_tot[warp] = v;
  }
  __syncthreads();
  if (tid < 256) {
    unsigned int above = 0;  // elements in the bins of higher warps
#pragma unroll
    for (int w = 1; w < 8; ++w) above += w > warp ? warp_tot[w] : 0;
    const unsigned int next = __shfl_down_sync(0xffffffffu, v, 1);
    const unsigned int S_d = v + above, S_next = lane == 31 ? above : next + above;  // S[d], S[d + 1]
    if (S_d >= remaining && S_next < remaining) {
      *s_prefix = prefix | ((uint32_t)tid << shift);
      *s_remaining = remaining - S_next;
      *s_count = S_d - S_next;
    }
  }
  __syncthreads();
  prefix = *s_prefix;
  remaining = *s_remaining;
  count = *s_count;
}

// Up to KPT x 1 024 candidates, which is every request of a few thousand tokens: a thread keeps the keys of KPT consecutive slots in
// registers, read once through shared memory.  With half_pool the keys are of the running maximum over the neighbouring candidates.
// Bound by the chain of block barriers, three per pass, hence: as soon as the bin of the k-th largest key holds TK_LIST keys or
// fewer, usually after two passes, these are listed and ranked by key and slot at once; consecutive slots make the emission one
// scan over threads and let neighbouring windows share their middle.  With four passes always, a window per key and a count per warp
// and round, the selection of 5 120 candidates at width 7 took 14 700 clocks: 1 050 for the loads, 2 600 the windows, 7 700 the
// passes, 2 650 the emission.  Back to back, before and now (us): 300 candidates 4.2 / 2.7, 900 4.1 / 2.6, 2 000 5.6 / 3.7, 3 000 5.8 / 4.7,
// 5 120 7.2 / 5.7, 8 192 9.2 / 8.3.  Windows, one layer's eviction of 8 192 slots, each slot's read by itself against neighbours in
// registers: width 3 17.5 / 15.9, width 7 19.3 / 16.3 (two heads); of 300 slots at width 853, walked whole against to the last candidate, 34.7 /
// 10.9.
constexpr int TK_LIST = 128;  // eight threads rank one key
template <int KPT>
__host__ __device__ constexpr int topk_at(int i) {  // place of slot i in shared memory: a thread's slots on banks of their own
  return KPT % 2 == 0 ? i + i / KPT : i;
}
template <int KPT>
__device__ __forceinline__ void topk_regs(const float* __restrict__ s, float* __restrict__ raw, int cand_begin, int n, int k, int half_pool,
                                          int32_t* __restrict__ idx_out, uint32_t* status) {
  __shared__ unsigned int whist[2][TK_HISTS][256];  // passes alternate: one is cleared while the other counts
  __shared__ unsigned int warp_tot[TK_WARPS];
  __shared__ unsigned int s_prefix, s_remaining, s_count, s_listed;
  __shared__ uint32_t list_key[TK_LIST], s_key;
  __shared__ int list_slot[TK_LIST], s_slot;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i0 = tid * KPT;
  float v[KPT];
#pragma unroll
  for (int j = 0; j < KPT; ++j) v[j] = tid + j * TK_THREADS < n ? __ldcg(s + tid + j * TK_THREADS) : 0.f;
  for (int i = tid; i < TK_HISTS * 256; i += TK_THREADS) (&whist[0][0][0])[i] = 0;
  if (tid == 0) s_listed = 0;
  if (KPT > 1 || half_pool > 0) {
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (tid + j * TK_THREADS < n) raw[topk_at<KPT>(tid + j * TK_THREADS)] = v[j];
    __syncthreads();
    const float none = __int_as_float(0x7fffffff);  // fmaxf passes over NaN
    auto get = [&](int i) { return i >= 0 && i < n ? raw[topk_at<KPT>(i)] : none; };
#pragma unroll
    for (int j = 0; j < KPT; ++j) v[j] = i0 + j < n ? raw[topk_at<KPT>(i0 + j)] : 0.f;
    if (2 * half_pool + 1 >= KPT && half_pool > 0) {
      // what all windows of the thread have in common, then what those before and those behind have besides
      float mid = none, run = none;
      const int m0 = max(0, i0 + KPT - 1 - half_pool), m1 = i0 < n ? min(n - 1, i0 + half_pool) : -1;
#pragma unroll 4
      for (int i = m0; i <= m1; ++i) mid = fmaxf(mid, raw[topk_at<KPT>(i)]);
#pragma unroll
      for (int j = KPT - 2; j >= 0; --j) {
        run = fmaxf(run, get(i0 + j - half_pool));
        v[j] = fmaxf(v[j], run);
      }
      run = mid;
#pragma unroll
      for (int j = 0; j < KPT; ++j) {
        if (j > 0) run = fmaxf(run, get(i0 + j + half_pool));
        v[j] = fmaxf(v[j], run);
      }
    } else if (half_pool > 0) {
      // windows narrower than the thread's slots: those and the few on either side, in registers
      constexpr int HM = KPT > 2 ? (KPT - 2) / 2 : 0;  // 2 half_pool + 1 < KPT
      float e[KPT + 2 * HM];
#pragma unroll
      for (int j = 0; j < KPT; ++j) e[HM + j] = i0 + j < n ? v[j] : none;
#pragma unroll
      for (int d = 1; d <= HM; ++d) {
        e[HM - d] = get(i0 - d);
        e[HM + KPT - 1 + d] = get(i0 + KPT - 1 + d);
      }
#pragma unroll
      for (int d = 1; d <= HM; ++d)
        if (d <= half_pool) {
#pragma unroll
          for (int j = 0; j < KPT; ++j) v[j] = fmaxf(v[j], fmaxf(e[HM + j - d], e[HM + j + d]));
        }
    }
  }
  uint32_t key[KPT];
  bool nonfinite = false;
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    nonfinite = nonfinite || (i0 + j < n && !(fabsf(v[j]) <= 3.0e38f));
    key[j] = score_key(v[j]);
  }
  if (nonfinite) atomicOr(status, A3_DEV_NONFINITE_SCORE);
  uint32_t prefix = 0, mask = 0;
  unsigned int remaining = (unsigned int)k, count = (unsigned int)n;  // keys with this prefix, and how many of them are taken
  __syncthreads();
#pragma unroll 1
  for (int pass = 0; pass < 4 && count > TK_LIST; ++pass) {
    const int shift = 24 - 8 * pass;
    unsigned int* mine = whist[pass & 1][warp % TK_HISTS];
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const bool in = i0 + j < n && (key[j] & mask) == prefix;
      if (!__any_sync(0xffffffffu, in)) continue;  // the rule behind the first passes
      const uint32_t digit = in ? (key[j] >> shift) & 255u : 0xFFFFFFFFu;
      const uint32_t first = __shfl_sync(0xffffffffu, digit, 0);
      if (__all_sync(0xffffffffu, digit == first)) {
        if (lane == 0) atomicAdd(&mine[digit], 32u);
      } else if (in) {
        atomicAdd(&mine[digit], 1u);
      }
    }
    for (int i = tid; i < TK_HISTS * 256; i += TK_THREADS) (&whist[(pass & 1) ^ 1][0][0])[i] = 0;
    __syncthreads();
    topk_bin(whist[pass & 1], warp_tot, &s_prefix, &s_remaining, &s_count, shift, prefix, remaining, count);
    mask |= 255u << shift;
  }
  // taken: keys above `prefix`, and of those equal to it the `remaining` lowest slots - or, listed, exactly those up to a key and slot
  const bool listed = count <= TK_LIST;
  if (listed) {
#pragma unroll
    for (int j = 0; j < KPT; ++j)
      if (i0 + j < n && (key[j] & mask) == prefix) {
        const unsigned int at = atomicAdd(&s_listed, 1u);
        list_key[at] = key[j];
        list_slot[at] = i0 + j;
      }
    __syncthreads();
    const unsigned int c = tid >> 3;  // 1 024 threads: TK_LIST keys
    unsigned int better = 0;
    const uint32_t my_key = c < count ? list_key[c] : 0;
    const int my_slot = c < count ? list_slot[c] : 0;
    for (unsigned int t = tid & 7; t < count; t += 8) better += list_key[t] > my_key || (list_key[t] == my_key && list_slot[t] < my_slot);
#pragma unroll
    for (int o = 4; o; o >>= 1) better += __shfl_xor_sync(0xffffffffu, better, o);
    if (c < count && better == remaining - 1 && (tid & 7) == 0) {
      s_key = my_key;
      s_slot = my_slot;
    }
    __syncthreads();
    prefix = s_key;
  }
  const int last_slot = listed ? s_slot : 0;
  // ordered emission: one scan of the counts, taken ones in the low half of the word and equal keys that wait for their turn in the high
  unsigned int mine = 0;
  bool gt[KPT], eq[KPT];
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const bool live = i0 + j < n;
    gt[j] = live && (key[j] > prefix || (listed && key[j] == prefix && i0 + j <= last_slot));
    eq[j] = live && !listed && key[j] == prefix;
    mine += (gt[j] ? 1u : 0u) + (eq[j] ? 0x10000u : 0u);
  }
  unsigned int upto = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int t = __shfl_up_sync(0xffffffffu, upto, o);
    if (lane >= o) upto += t;
  }
  if (lane == 31) warp_tot[warp] = upto;
  __syncthreads();
  const unsigned int before = upto - mine + __reduce_add_sync(0xffffffffu, lane < warp ? warp_tot[lane] : 0u);
  unsigned int my_gt = before & 0xFFFFu, my_eq = before >> 16;
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    if (gt[j] || (eq[j] && my_eq < remaining)) {
      const unsigned int o = my_gt + (my_eq < remaining ? my_eq : remaining);
      if (o < (unsigned int)k) idx_out[o] = cand_begin + i0 + j;
    }
    my_gt += gt[j] ? 1 : 0;
    my_eq += eq[j] ? 1 : 0;
  }
}

template <bool IN_SMEM>
__device__ __forceinline__ void topk_body(const float* __restrict__ s, uint32_t* __restrict__ keys, int cand_begin, int n, int k,
                                          int32_t* __restrict__ idx_out, uint32_t* status) {
  __shared__ unsigned int whist[TK_HISTS][256];
  __shared__ unsigned int warp_tot[8];
  __shared__ unsigned int s_prefix, s_remaining, s_count;
  __shared__ unsigned int warp_gt[TK_WARPS], warp_eq[TK_WARPS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // past L1: this CTA may have become resident while the kernel that writes the scores was still running
  auto key_at = [&](int i) -> uint32_t { return IN_SMEM ? keys[i] : score_key(__ldcg(s + i)); };

  // ---- load: scores -> keys (shared memory), non-finite scores flagged
  bool nonfinite = false;
#pragma unroll 4
  for (int i = tid; i < n; i += TK_THREADS) {
    const float v = __ldcg(s + i);
    if (!(fabsf(v) <= 3.0e38f)) nonfinite = true;
    if (IN_SMEM) keys[i] = score_key(v);
  }
  if (nonfinite) atomicOr(status, A3_DEV_NONFINITE_SCORE);

  // ---- radix select: after the loop `prefix` is the key of the k-th largest element
  uint32_t prefix = 0, mask = 0;
  unsigned int count;
  unsigned int remaining = (unsigned int)k;  // rank (1-based, from the top) inside the current bucket
  const int n_round = (n + 31) & ~31;        // whole warps walk the array, so that the lanes can vote together
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int i = tid; i < TK_HISTS * 256; i += TK_THREADS) (&whist[0][0])[i] = 0;
    __syncthreads();
    unsigned int* mine = whist[warp % TK_HISTS];
    for (int i = tid; i < n_round; i += TK_THREADS) {
      uint32_t digit = 0xFFFFFFFFu;  // lanes with nothing to count
      if (i < n) {
        const uint32_t key = key_at(i);
        if ((key & mask) == prefix) digit = (key >> shift) & 255u;
      }
      const uint32_t first = __shfl_sync(0xffffffffu, digit, 0);
      if (__all_sync(0xffffffffu, digit == first)) {
        if (lane == 0 && digit != 0xFFFFFFFFu) atomicAdd(&mine[digit], 32u);
      } else if (digit != 0xFFFFFFFFu) {
        atomicAdd(&mine[digit], 1u);
      }
    }
    __syncthreads();
    topk_bin(whist, warp_tot, &s_prefix, &s_remaining, &s_count, shift, prefix, remaining, count);
    mask |= 255u << shift;
  }
  // `remaining` = how many elements equal to the threshold key are taken (lowest slots first)
  const uint32_t thr = prefix;
  const unsigned int need_eq = remaining;

  // ---- ordered emission: warp w owns slots [w * span, (w + 1) * span)
  const int span = ((n + TK_WARPS - 1) / TK_WARPS + 31) & ~31;
  const int b0 = warp * span, b1 = min(n, b0 + span);
  unsigned int cnt_gt = 0, cnt_eq = 0;
  for (int base = b0; base < b1; base += 32) {
    const int i = base + lane;
    const uint32_t key = i < b1 ? key_at(i) : 0u;
    cnt_gt += __popc(__ballot_sync(0xffffffffu, i < b1 && key > thr));
    cnt_eq += __popc(__ballot_sync(0xffffffffu, i < b1 && key == thr));
  }
  if (lane == 0) {
    warp_gt[warp] = cnt_gt;
    warp_eq[warp] = cnt_eq;
  }
  __syncthreads();
  unsigned int run_gt = 0, run_eq = 0;
  for (int w = 0; w < warp; ++w) {
    run_gt += warp_gt[w];
    run_eq += warp_eq[w];
  }
  const unsigned int lt_mask = (1u << lane) - 1u;
  for (int base = b0; base < b1; base += 32) {
    const int i = base + lane;
    const uint32_t key = i < b1 ? key_at(i) : 0u;
    const bool gt = i < b1 && key > thr, eq = i < b1 && key == thr;
    const unsigned int bgt = __ballot_sync(0xffffffffu, gt), beq = __ballot_sync(0xffffffffu, eq);
    const unsigned int my_gt = run_gt + __popc(bgt & lt_mask);  // greater-than elements before me
    const unsigned int my_eq = run_eq + __popc(beq & lt_mask);  // equal elements before me
    if (gt || (eq && my_eq < need_eq)) {
      const unsigned int o = my_gt + (my_eq < need_eq ? my_eq : need_eq);
      if (o < (unsigned int)k) idx_out[o] = cand_begin + i;
    }
    run_gt += __popc(bgt);
    run_eq += __popc(beq);
  }
}

// REGS > 0: at most REGS x 1 024 candidates, in registers; 0: any number, in shared memory or re-read from global memory
template <int REGS>
__global__ void __launch_bounds__(TK_THREADS)
topk_select_kernel(const float* __restrict__ scores, int cand_begin, int n, int k, int32_t* __restrict__ idx_out, uint32_t* status,
                   size_t score_stride, size_t idx_stride, int in_smem, int half_pool, int tail_begin, int tail) {
  extern __shared__ uint32_t tk_keys[];
  pdl_wait();
  pdl_launch_dependents();
  // one CTA per independent selection (the per-head selections of the eviction step; a single one for Eq. 3)
  const float* s = scores + blockIdx.x * score_stride + cand_begin;
  int32_t* out = idx_out + blockIdx.x * idx_stride;
  for (int i = threadIdx.x; i < tail; i += TK_THREADS) out[k + i] = tail_begin + i;
  if constexpr (REGS > 0) {
    topk_regs<REGS>(s, reinterpret_cast<float*>(tk_keys), cand_begin, n, k, half_pool, out, status);
    return;
  }
  if (in_smem) topk_body<true>(s, tk_keys, cand_begin, n, k, out, status);
  else topk_body<false>(s, tk_keys, cand_begin, n, k, out, status);
}

static int launch_topk(const a3_handle* h, const float* scores, size_t score_stride, int batches, int cand_begin, int n, int k,
                       int half_pool, int tail_begin, int tail, int32_t* idx_out, size_t idx_stride, cudaStream_t st) {
  const int in_smem = n <= TK_SMEM_KEYS ? 1 : 0;
  ProfScope prof(h, A3_K_TOPK, st);
  auto go = [&](auto kernel, size_t smem) {
    return launch_pdl(kernel, dim3(batches), dim3(TK_THREADS), smem, st, scores, cand_begin, n, k, idx_out, h->dev_status, score_stride, idx_stride,
                      in_smem, half_pool, tail_begin, tail);
  };
  // Time grows with the keys per thread (back to back 900 candidates 2.6 us, 3 000 4.7, 5 120 5.7, 8 192 8.3), hence instances of one,
  // three, five and eight: the smallest that holds the candidates.  Those in between would save 0.4 us (2 000 candidates 4.4 / 4.0, 4 000
  // 5.9 / 5.6), 1.0 (6 000 8.1 / 7.1) and 0.6 (7 000 8.2 / 7.7) and are left out.
  if (n <= TK_THREADS) {
    A3_CUDA(go(topk_select_kernel<1>, half_pool > 0 ? (size_t)n * 4 : 0));
  } else if (n <= 3 * TK_THREADS) {
    A3_CUDA(go(topk_select_kernel<3>, (size_t)n * 4));
  } else if (n <= 5 * TK_THREADS) {
    static SmemAttrOnce attr5;
    A3_TRY(smem_attr_once(attr5, h->device, topk_select_kernel<5>, 5 * TK_THREADS * 4));
    A3_CUDA(go(topk_select_kernel<5>, (size_t)n * 4));
  } else if (n <= 8 * TK_THREADS) {
    static SmemAttrOnce attr8;
    A3_TRY(smem_attr_once(attr8, h->device, topk_select_kernel<8>, topk_at<8>(8 * TK_THREADS) * 4));
    A3_CUDA(go(topk_select_kernel<8>, (size_t)topk_at<8>(n) * 4));
  } else {
    static SmemAttrOnce attr;
    A3_TRY(smem_attr_once(attr, h->device, topk_select_kernel<0>, TK_SMEM_KEYS * 4));
    A3_CUDA(go(topk_select_kernel<0>, in_smem ? (size_t)n * 4 : 0));
  }
  A3_LAUNCHED();
  return A3_OK;
}

}  // namespace a3

using namespace a3;

extern "C" int a3_topk_select(const a3_handle* h, const float* scores, int cand_begin, int cand_end, int k,
                              int32_t* idx_out, a3_stream stream) {
  if (!h || cand_begin < 0 || cand_end < cand_begin || k < 0) return A3_EINVAL;
  const int n = cand_end - cand_begin;
  if (k > n) k = n;
  if (k == 0) return A3_OK;
  if (!scores || !idx_out) return A3_EINVAL;
  return launch_topk(h, scores, 0, 1, cand_begin, n, k, 0, 0, 0, idx_out, 0, (cudaStream_t)stream);
}

int a3::topk_rows(const a3_handle* h, const float* scores, int cand_begin, int cand_end, int k, int tail_begin, int tail, int32_t* idx_out,
                  cudaStream_t st) {
  if (k <= 0) return iota_rows(h, idx_out, tail_begin, tail, st);
  return launch_topk(h, scores, 0, 1, cand_begin, cand_end - cand_begin, k, 0, tail_begin, tail, idx_out, 0, st);
}

// Pooling inside the selection saves a launch (2.5 us) and costs every thread its windows in shared-memory reads, in the one CTA of a
// head where the kernel of its own has the whole chip.  One layer's eviction, votes to gather, inside / apart (us; Llama-8B heads, two
// heads).  On this side of the line: 300 candidates at width 255 11.7 / 13.8 and 10.7 / 12.7, 900 at 283 14.6 / 16.7 and 13.4 / 14.4, 1 024
// at 249 14.3 / 15.2 and 13.3 / 13.9, 2 000 at 127 15.1 / 17.0 and 12.6 / 13.8, 5 120 at 7 16.2 / 17.5 and 12.7 / 14.0, at 49 17.2 / 18.1 and
// 13.6 / 14.7, 8 192 at 7 20.6 / 21.9 and 15.9 / 17.5, at 31 22.0 / 22.9 and 16.7 / 17.6.  Beyond it inside has become the faster side too
// since windows share their middle: 1 024 at 251 14.3 / 15.2 and 13.4 / 14.0, 2 000 at 191 14.1 / 16.4 and 13.1 / 14.2, 5 120 at 129 18.3 / 19.3
// and 15.0 / 15.9, 8 192 at 63 23.1 / 23.7 and 18.5 / 19.2; the line stays where it was drawn against a window per key, and where
// tests/test_gpu_evict.py counts launches on either side.  Candidates that do not fit the registers would read their window from global
// memory, which loses at every width (32 768 79.1 / 70.9 at 7, 215 / 82 at 255).
bool a3::topk_can_pool(int n_cand, int pool) { return n_cand <= 8 * TK_THREADS && (long long)n_cand * pool <= 250 * TK_THREADS; }

int a3::topk_batched(const a3_handle* h, const float* scores, size_t score_stride, int batches, int cand_begin, int cand_end,
                     int k, int pool, int32_t* idx_out, size_t idx_stride, cudaStream_t st) {
  const int n = cand_end - cand_begin;
  if (k > n) k = n;
  if (k <= 0 || batches <= 0) return A3_OK;
  return launch_topk(h, scores, score_stride, batches, cand_begin, n, k, pool > 1 ? pool / 2 : 0, 0, 0, idx_out, idx_stride, st);
}
