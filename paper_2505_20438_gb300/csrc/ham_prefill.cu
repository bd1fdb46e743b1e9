// Chunked prefill over the paged smashed-KV cache (sm_103a): prompt ingestion.
//
// What it computes (HAMburger, arXiv 2505.20438): only response tokens are fused into
// multi-token slots (Figure 2, training), so a prompt's tokens each become one slot, stored
// exactly as the decode path's append stores a slot (RoPE at the slot's position, Sec. 3.2;
// one KV set per slot, Sec. 3.1).  The chunk's queries then attend causally: new row j of a
// sequence holding L slots attends over slots 0 .. L + j (Llama-3.2 base model, Sec. 4.1:
// softmax scale 1/sqrt(d), query head h reads KV head h / G).  Unlike decode this is a dense
// contraction: every K/V tile serves 128 query rows, so it runs on the tensor cores.
//
// Three launches (four when the attention splits over the cached slots):
//  1. prefill_plan_kernel, one block per sequence: checks that the sequence's rows fit
//     (counts, capacity, pages), gives each row its position (slot index, running token count
//     or the caller's) and pool row (or -1: not stored), orders the query blocks, and advances the
//     token count.
//  2. prefill_rope_kernel, one block per row: turns q and k at the row's position and stores
//     k and v into the row's slot.  The rotation x0 c - x1 s is evaluated from the fp64 cos/sin
//     table in pairs of fp32 values (error-free products and sums, about 48 bits) and rounded
//     once to bf16, which gives the bits of the fp64 evaluation except when the exact value
//     lies within ~2^-44 (relative) of a rounding boundary.  This GPU's fp64 pipe would take
//     about half a millisecond for a 16k-row chunk of a Llama-8B layer; the fp32 pairs take
//     microseconds.
//  3. prefill_attn_kernel, a persistent grid (one CTA an SM) over items of one KV head and two Q
//     tiles of 128 (query row, head) rows of one sequence: S = Q K^T and O += P V on the
//     5th-generation tensor cores (tcgen05.mma kind::f16, M = 128, bf16 operands, fp32 accumulators
//     in tensor memory).  Q, K and V reach shared memory by TMA (128-slot K/V tiles of eight
//     16-slot chunks, one box each, in one ring; two producer warps look the pages up 32 chunks
//     ahead).  A warp for each Q tile issues its products; eight softmax warps, one thread a row,
//     read S from tensor memory, keep the online softmax in fp32 (exp2 domain, running maximum
//     raised only past 2^8), write the bf16 probabilities over the scores (the A operand of
//     O += P V) and rescale O in tensor memory when the maximum moves.  The causal mask applies to
//     the blocks that reach past a row's own slot; items are handed out from a counter in the
//     plan's order, the blocks that attend over the most slots first.
//     When the items would leave SMs idle (a short chunk: few query blocks) they are split over
//     slots: a sequence with L cached slots is cut into up to floor(L / 512) contiguous ranges
//     of 128-slot tiles (the last range also takes the chunk's own slots), and a split that is
//     not alone leaves its rows' unnormalised output, running maximum and sum as a partial.
//     Bound by each Q tile's chain scores -> softmax -> P V -> scores, which the other tile's
//     covers in part: the tensor pipe is about 60% busy.  The whole call, in a loop of calls on one set
//     of buffers (with buffers that change from call to call 2% more): 4 fresh prompts x 4096 rows
//     of a Llama-8B layer 477 us, against 565 with 64-slot tiles, four issuing warps whose operands
//     sat in per-thread registers and a CTA an item; 64 rows over 65,536 slots 80 against 142 us (with
//     the merge below); 4 x 2048 rows over 2048 slots at head_dim 64 263 against 345; 256 prompts of
//     32 rows 102 against 175.
//  4. prefill_merge_kernel (split launches only), one warp per (row, head): the split-softmax
//     merge of the partials in split order (as the decode combine merges its CTAs').
//
// Every wait is bounded (about 2 s); a wait that runs out records HAM_DEVERR_TIMEOUT, lets the
// CTA's copies land and returns.  No trap, no unbounded spin.
#include <cuda.h>
#include <cuda_bf16.h>

#include <cmath>
#include <type_traits>

#include "ham_internal.cuh"
#include "ham_order.cuh"
#include "ham_prefill.cuh"
#include "ham_ptx.cuh"
#include "ham_turns.cuh"

namespace ham {
namespace {

constexpr int kPlanThreads = 256;
constexpr int kPlanRun = 8;  // consecutive rows a plan thread takes per tile
constexpr float kRescaleSlack = 8.0f;  // log2 units: the running max lags by at most 2^8
constexpr int kRopeThreads = 384;  // at most

// ------------------------------------------------------------------------------------
// 1. plan
// ------------------------------------------------------------------------------------
__device__ __forceinline__ int block_sum(int x, int *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
  __syncthreads();  // red may still be read from a previous call
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  int total = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) total += red[w];
  return total;
}

// Inclusive prefix sum over the block (thread order); *total gets the block's sum.
__device__ __forceinline__ int block_scan(int x, int *red, int *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();
  if (lane == 31) red[warp] = x;
  __syncthreads();
  int before = 0, all = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    if (w < warp) before += red[w];
    all += red[w];
  }
  *total = all;
  return x + before;
}

__global__ void __launch_bounds__(kPlanThreads) prefill_plan_kernel(PrefillView v, int qb_shift) {
  __shared__ int red[kPlanThreads / 32];
  const int b = blockIdx.x, tid = threadIdx.x, B = v.batch;
  // The RoPE kernel may be scheduled now: it reads the call's inputs, and waits for this grid (which
  // itself starts after everything before it on the stream) before it reads the plan or writes.
  grid_launch_dependents();
  if (b == 0 && tid == 0) *v.next_item = 0;  // the attention's items are handed out from here
  // The offsets must describe the call's rows: every block checks all of them, so that all agree.
  int bad_off = 0;
  for (int i = tid; i < B; i += kPlanThreads) bad_off |= v.offsets[i + 1] < v.offsets[i];
  if (tid == 0) bad_off |= v.offsets[0] != 0 || v.offsets[B] != v.rows;
  bad_off = __syncthreads_or(bad_off);
  if (bad_off) {
    if (tid == 0) {
      v.seq_info[b] = make_int4(-1, 0, 0, 0);
      if (b == 0) {
        v.next_item[1] = 0;  // no query blocks
        record_error(v.err, HAM_DEVERR_NTOK);
      }
    }
    return;
  }
  const int a = v.offsets[b], n = v.offsets[b + 1] - a;
  const int L = v.num_slots[b];
  // The order of the query blocks in the attention (ham_order.cuh): the place of each of this
  // sequence's, by a group of 2^g threads that share the other sequences.  The counters do not change
  // while the plan runs: the attention, which starts after all of it, advances num_slots.
  auto slots_of = [&](int c) { return (uint32_t)max(0, min(v.num_slots[c], v.max_slots)); };
  {
    const int g = B >= 32 ? 5 : 32 - __clz(B - 1);  // (B = 1: 0)
    const int m = (int)query_blocks(n, qb_shift), share = tid & ((1 << g) - 1);
    const uint32_t own = slots_of(b);
    for (int j0 = 0; j0 < m; j0 += kPlanThreads >> g) {  // (the same trip count in every thread)
      const int j = j0 + (tid >> g);
      const uint32_t reach = block_reach(own, n, j, qb_shift);
      uint32_t at = 0;
      if (j < m) {
        for (int c = share; c < B; c += 1 << g)
          if (c != b)
            at += blocks_before(slots_of(c), v.offsets[c + 1] - v.offsets[c], reach, c < b, qb_shift);
      }
      for (int o = 1; o < 1 << g; o <<= 1) at += __shfl_xor_sync(kFull, at, o);
      if (j < m && share == 0) v.order[at + (m - 1 - j)] = make_int2(b, j);
    }
  }
  if (b == 0) {
    int m = 0;
    for (int c = tid; c < B; c += kPlanThreads) m += query_blocks(v.offsets[c + 1] - v.offsets[c], qb_shift);
    m = block_sum(m, red);
    if (tid == 0) v.next_item[1] = m;
  }
  int err = 0;
  if (L < 0 || L > v.max_slots) err = HAM_DEVERR_SLOTS;
  else if ((int64_t)L + n > v.max_slots) err = HAM_DEVERR_CAPACITY;
  int bad_tok = 0, bad_page = 0;
  if (!err && n > 0) {
    if (v.ntok)
      for (int j = tid; j < n; j += kPlanThreads) bad_tok |= v.ntok[a + j] < 1;
    const int p0 = L / v.page_slots, p1 = (L + n - 1) / v.page_slots;
    for (int pg = p0 + tid; pg <= p1; pg += kPlanThreads) {
      const int page = v.page_table[(int64_t)b * v.max_pages + pg];
      bad_page |= page < 0 || page >= v.pool_pages;
    }
  }
  bad_tok = __syncthreads_or(bad_tok);
  bad_page = __syncthreads_or(bad_page);
  if (!err && bad_tok) err = HAM_DEVERR_NTOK;
  if (!err && bad_page) err = HAM_DEVERR_PAGE;
  if (err) {  // none of the rows is stored
    for (int j = tid; j < n; j += kPlanThreads) v.row_info[a + j] = make_int2(0, -1);
    if (tid == 0) {
      record_error(v.err, err);
      v.seq_info[b] = make_int4(-1, n, a, 1);
    }
    return;
  }
  // positions (the caller's, the slot index, or the tokens before the row) and pool rows.  A
  // thread takes kPlanRun consecutive rows of each tile of kPlanThreads * kPlanRun rows: their
  // token counts, positions and page-table entries are loaded together, and one block scan of
  // the threads' sums a tile gives every row its tokens before it.
  const int64_t t0 = v.num_tokens[b];
  int64_t carry = 0;
  for (int j0 = 0; j0 < n; j0 += kPlanThreads * kPlanRun) {
    const int jb = j0 + tid * kPlanRun;
    int t[kPlanRun], run = 0;
#pragma unroll
    for (int k = 0; k < kPlanRun; ++k) {
      t[k] = jb + k < n ? (v.ntok ? v.ntok[a + jb + k] : 1) : 0;
      run += t[k];
    }
    int total = 0;
    int64_t before = t0 + carry + (block_scan(run, red, &total) - run);
#pragma unroll
    for (int k = 0; k < kPlanRun; ++k) {
      const int j = jb + k;
      if (j < n) {
        int64_t p;
        if (v.pos) p = v.pos[a + j];
        else if (v.pos_mode == HAM_POS_SLOT) p = (int64_t)L + j;
        else p = before;
        const int slot = L + j, pg = slot / v.page_slots;
        const int page = v.page_table[(int64_t)b * v.max_pages + pg];
        v.row_info[a + j] = make_int2((int32_t)p, page * v.page_slots + (slot - pg * v.page_slots));
      }
      before += t[k];
    }
    carry += total;
  }
  if (tid == 0) {
    v.seq_info[b] = make_int4(L, n, a, 1);
    v.num_tokens[b] = t0 + carry;
  }
}

// ------------------------------------------------------------------------------------
// 2. RoPE + append
// ------------------------------------------------------------------------------------
// bf16 bits of hi + lo (|lo| <= half an fp32 ulp of hi), rounded to nearest, ties to even:
// the rounding of hi alone, except where hi sits exactly halfway between two bf16 values and
// lo says on which side the sum lies.
__device__ __forceinline__ uint16_t bf16_of_pair(float hi, float lo) {
  const uint32_t u = __float_as_uint(hi);
  if ((u & 0xFFFFu) == 0x8000u && lo != 0.f && (u & 0x7F800000u) != 0x7F800000u) {
    const bool away = (lo > 0.f) == (hi > 0.f);
    return (uint16_t)((u >> 16) + (away ? 1u : 0u));
  }
  return __bfloat16_as_ushort(__float2bfloat16_rn(hi));
}

// Fast evaluation of a c - b s, with c = ch + cl and s = sh + sl given as fp32 pairs and a, b
// exact (bf16 values): y = a ch - b sh in plain fp32 lies within 3 * 2^-24 (|a| + |b|) < e / 2
// of the exact value, e = (|a| + |b|) 2^-21.  When no bf16 rounding boundary is within e of y
// (the nearest one is the midpoint sharing y's upper 16 bits; the others are a quarter of a
// bf16 spacing away, more than e once e < 2^-11 |y|), the exact value rounds as y does and
// *sure is set; otherwise rotate_exact gives the rounding.
__device__ __forceinline__ float rotate_fast(float a, float b, float ch, float sh, float e,
                                             bool *sure) {
  const float y = __fmaf_rn(a, ch, -__fmul_rn(b, sh));
  const float mid = __uint_as_float((__float_as_uint(y) & 0xFFFF0000u) | 0x8000u);
  *sure = fabsf(__fsub_rn(y, mid)) > e && e < __fmul_rn(fabsf(y), 0x1p-11f);
  return y;
}

// a c - b s rounded once to bf16 near a rounding boundary: products by FMA error terms and sums
// by two-sum are exact, only the small terms are rounded, so the pair carries about 48 bits of
// the exact value.
__device__ __noinline__ uint16_t rotate_exact(float a, float b, float ch, float cl, float sh,
                                              float sl) {
  const float p1 = __fmul_rn(a, ch), e1 = __fmaf_rn(a, ch, -p1);
  const float p2 = __fmul_rn(b, sh), e2 = __fmaf_rn(b, sh, -p2);
  const float s = __fsub_rn(p1, p2);  // two-sum of p1 and -p2: s + t = p1 - p2
  const float bp = __fsub_rn(s, p1);
  const float t = __fadd_rn(__fsub_rn(p1, __fsub_rn(s, bp)), __fsub_rn(-p2, bp));
  const float low =
      __fmaf_rn(a, cl, __fmaf_rn(-b, sl, __fadd_rn(t, __fsub_rn(e1, e2))));
  if (low == 0.f) return __bfloat16_as_ushort(__float2bfloat16_rn(s));  // keeps s's zero sign
  const float hi = __fadd_rn(s, low);  // two-sum of s and low
  const float hb = __fsub_rn(hi, s);
  const float lo = __fadd_rn(__fsub_rn(s, __fsub_rn(hi, hb)), __fsub_rn(low, hb));
  return bf16_of_pair(hi, lo);
}

__device__ __forceinline__ float bf16_value(uint16_t b) {
  return __uint_as_float((uint32_t)b << 16);
}

__device__ __forceinline__ void split_double(double x, float &hi, float &lo) {
  hi = __double2float_rn(x);
  lo = __double2float_rn(x - (double)hi);  // x - hi is exact in fp64
}

// Shared-memory index of frequency i of the (cos, sin) row: the eight frequencies a thread
// reads, 8 (i / 8) .. + 7, rotated by i / 8 within their group of eight, so that the eight
// threads of a head (distinct i / 8, same step) read eight distinct 16-byte bank groups.
__device__ __forceinline__ int cs_index(int i) { return (i & ~7) | ((i + (i >> 3)) & 7); }

// One block per row.  Thread t owns the eight pairs (i, i + d/2), i = 8 (t % (d/16)) .. + 7, of
// heads t / (d/16), t / (d/16) + threads / (d/16), ... (query heads, then key heads): a 16-byte load
// and store of each half.  The block is as large as the row's heads ask for, up to kRopeThreads, so
// that the usual rows take one pass (kMore: more than one): a block's time is its chain of loads and
// one rotation, and rows in flight are what covers it.  Held at the registers of five blocks of
// kRopeThreads (six of 320 threads are resident).  The whole call in a loop, before the later changes
// of the attention: 4 x 4096 rows of 40 heads 482 us, 491 at four, 508 at three, 487 with blocks of 256
// threads in two uneven passes; 2 x 4096 rows of 16 heads 88.6 and 96.2; 4 x 2048 rows at head_dim 64
// 262.8 and 270.7.  The plan left the row's position and pool row in row_info, so every load the block
// makes needs only the row index, and is issued at once: the first two heads' halves, a 16-byte piece
// of the value row, and then the (cos, sin) row of the position, which goes to shared memory, read by
// the threads of every head.
template <int D, typename OutT, bool kMore>
__global__ void __launch_bounds__(kRopeThreads, kMore ? 3 : 5) prefill_rope_kernel(PrefillView v) {
  constexpr int kHalf = D / 2, kOcts = kHalf / 8;
  const int threads = blockDim.x, heads_pass = threads / kOcts;
  constexpr int kVPieces = D / 8;  // 16-byte pieces of one head's value row
  static_assert(kHalf <= kRopeThreads, "one thread a frequency");
  __shared__ float4 cs_s[kHalf];   // (c_hi, c_lo, s_hi, s_lo) of frequency i at cs_index(i)
  const int64_t r = blockIdx.x;
  const int tid = threadIdx.x, j = tid % kOcts, h0 = tid / kOcts, h1 = h0 + heads_pass;
  const int Hq = v.n_q_heads, Hkv = v.n_kv_heads, H = Hq + Hkv, nv = Hkv * kVPieces;
  uint16_t *const qrow = v.q + r * Hq * D;
  const uint16_t *const krow = v.k_new + r * Hkv * D;
  const uint4 *const vrow = reinterpret_cast<const uint4 *>(v.v_new + r * Hkv * D);
  auto half_of = [&](int h, int upper) {  // 16-byte piece j of head h's lower or upper half
    const uint16_t *src = h < Hq ? qrow + h * D : krow + (h - Hq) * D;
    return *reinterpret_cast<const uint4 *>(src + upper * kHalf + 8 * j);
  };
  // 1. the loads: the call's inputs, then what the plan left (the row's pool row is -1 when it is
  //    not stored; the call's offsets are valid when sequence 0's plan entry says so)
  uint4 x0l{}, x0h{}, x1l{}, x1h{}, vv{};
  if (h0 < H) { x0l = half_of(h0, 0); x0h = half_of(h0, 1); }
  if (kMore && h1 < H) { x1l = half_of(h1, 0); x1h = half_of(h1, 1); }
  if (tid < nv) vv = vrow[tid];
  grid_dependency_wait();
  grid_launch_dependents();  // the attention may be scheduled as this grid drains
  const int2 ri = v.row_info[r];
  const int offsets_ok = v.seq_info[0].w;
  const int p = ri.x;
  const bool in_table = p >= 0 && p < v.rope_positions;
  float4 c4{};
  if (tid < kHalf && in_table) c4 = v.rope_table_ff[(int64_t)p * kHalf + tid];
  if (!offsets_ok || ri.y < 0) {  // not stored: its output rows are 0
    OutT *o = static_cast<OutT *>(v.out) + r * Hq * D;
    for (int e = tid; e < Hq * D; e += threads) o[e] = OutT(0.f);
    return;
  }
  // 2. the (cos, sin) row in shared memory (past the table: from fp64 sincos) and the slot's
  //    page and row in it
  __shared__ int2 where;  // (page, row in page)
  if (tid < kHalf) {
    if (!in_table) {
      double c, sn;
      sincos((double)p * v.inv_freq[tid], &sn, &c);
      split_double(c, c4.x, c4.y);
      split_double(sn, c4.z, c4.w);
    }
    cs_s[cs_index(tid)] = c4;
  }
  if (tid == 0) {
    where = make_int2(ri.y / v.page_slots, ri.y % v.page_slots);
    v.slot_pos[ri.y] = p;
    v.slot_ntok[ri.y] = v.ntok ? v.ntok[r] : 1;
  }
  __syncthreads();
  const int64_t page = where.x;
  const int prow = where.y;
  auto pool_row = [&](uint16_t *pool, int g) {
    return pool + ((page * Hkv + g) * v.page_slots + prow) * D;
  };
  // 3. the value row (a bit copy)
  if (tid < nv) reinterpret_cast<uint4 *>(pool_row(v.v_pool, tid / kVPieces))[tid % kVPieces] = vv;
  for (int e = tid + threads; e < nv; e += threads)
    reinterpret_cast<uint4 *>(pool_row(v.v_pool, e / kVPieces))[e % kVPieces] = vrow[e];
  // 4. query heads in place, key heads into the slot
  // Every output by the fast path, two to a conversion; the rare outputs whose rounding the
  // fast path leaves open (bit 2 m + u of `open`: pair m, lower (u = 0) or upper half) are
  // redone exactly in a loop of their own, so the exact path costs nothing where it is not used.
  auto rotate_store = [&](int h, const uint4 &xl, const uint4 &xh) {
    uint16_t *dst = h < Hq ? qrow + h * D : pool_row(v.k_pool, h - Hq);
    uint32_t wl[4] = {xl.x, xl.y, xl.z, xl.w}, wh[4] = {xh.x, xh.y, xh.z, xh.w};
    uint32_t open = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float yl[2], yh[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float4 c = cs_s[cs_index(8 * j + 2 * k + e)];
        const float x0 = bf16_value((uint16_t)(wl[k] >> (16 * e)));
        const float x1 = bf16_value((uint16_t)(wh[k] >> (16 * e)));
        const float err = __fmul_rn(__fadd_rn(fabsf(x0), fabsf(x1)), 0x1p-21f);
        bool sure_l, sure_h;
        yl[e] = rotate_fast(x0, x1, c.x, c.z, err, &sure_l);   // x0 c - x1 s
        yh[e] = rotate_fast(x1, x0, c.x, -c.z, err, &sure_h);  // x1 c + x0 s
        open |= (sure_l ? 0u : 1u) << (2 * (2 * k + e));
        open |= (sure_h ? 0u : 2u) << (2 * (2 * k + e));
      }
      const __nv_bfloat162 ol = __floats2bfloat162_rn(yl[0], yl[1]);
      const __nv_bfloat162 oh = __floats2bfloat162_rn(yh[0], yh[1]);
      const uint32_t uol = *reinterpret_cast<const uint32_t *>(&ol);
      const uint32_t uoh = *reinterpret_cast<const uint32_t *>(&oh);
      wl[k] = uol;  // wl/wh now hold outputs; the exact path reads the inputs from xl/xh
      wh[k] = uoh;
    }
    while (open) {
      const int bit = __ffs(open) - 1;
      open &= open - 1;
      const int m = bit >> 1, k = m >> 1, e = m & 1, upper = bit & 1;
      const uint32_t in_l = k == 0 ? xl.x : k == 1 ? xl.y : k == 2 ? xl.z : xl.w;
      const uint32_t in_h = k == 0 ? xh.x : k == 1 ? xh.y : k == 2 ? xh.z : xh.w;
      const float4 c = cs_s[cs_index(8 * j + m)];
      const float x0 = bf16_value((uint16_t)(in_l >> (16 * e)));
      const float x1 = bf16_value((uint16_t)(in_h >> (16 * e)));
      const uint32_t y = upper ? rotate_exact(x1, x0, c.x, c.y, -c.z, -c.w)
                               : rotate_exact(x0, x1, c.x, c.y, c.z, c.w);
      const uint32_t keep = e ? 0x0000FFFFu : 0xFFFF0000u, put = y << (16 * e);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        if (kk != k) continue;
        if (upper) wh[kk] = (wh[kk] & keep) | put;
        else wl[kk] = (wl[kk] & keep) | put;
      }
    }
    *reinterpret_cast<uint4 *>(dst + 8 * j) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
    *reinterpret_cast<uint4 *>(dst + kHalf + 8 * j) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
  };
  if (h0 < H) rotate_store(h0, x0l, x0h);
  if constexpr (kMore) {
    if (h1 < H) rotate_store(h1, x1l, x1h);
    for (int h = h1 + heads_pass; h < H; h += heads_pass)
      rotate_store(h, half_of(h, 0), half_of(h, 1));
  }
}

// ------------------------------------------------------------------------------------
// 3. causal attention of the chunk, on the 5th-generation tensor cores (tcgen05)
// ------------------------------------------------------------------------------------
// A work item is one KV head, two Q tiles of 128 rows each and (split launches) one range of
// slots; a row is a (query row, head) pair, m = (row - first row of the tile) * G + head within
// the group, and sits in TMEM lane m.  CTAs (one an SM) take items from a counter, the blocks that
// attend over the most slots first; an item's last softmax and output run beside the next one's
// first copies.
//
// K and V come in tiles of 128 slots; the softmax works on blocks of 64 (half tiles).  Tensor-memory
// columns per Q tile q: two blocks of scores S_q (64 fp32 each; the first 32 columns of a block then
// hold its probabilities P, bf16 pairs, the A operand of O += P V) and O_q (head_dim fp32).  One
// thread a Q tile issues its products: O += P V of a block, then the S whose columns that frees.
// Nothing but the order of issue says that P V has read P when S overwrites it.  PTX promises that order
// for products on one accumulator; these two have different ones (P is an operand of the first and lies
// in the columns that the second writes), so the kernel relies on the tensor core taking the products
// of one thread in the order in which it issued them, whatever their accumulators.  A wait for P V before
// S gives the same bits and costs 1 to 6% (4 x 4096 rows 507 us and 489, ragged chunks 247 and 233, 64
// rows over 65,536 slots 81.7 and 80.6).
//  - head_dim 128: S of a tile (N = 128) follows P V of the second block of the tile before.  While
//    the products of one Q tile run, the other's softmax does: the two softmax groups take turns,
//    tile by tile.  (Left to themselves they fall into step, compete for the issue slots and then
//    for the tensor cores: 6% slower.  With S in blocks, N = 64, a product takes the 64 cycles of
//    N = 128, bound by the shared-memory reads of Q: also slower.)
//  - head_dim 64: half the products for the same softmax, which bounds it: S of a block (N = 64) is
//    two blocks ahead and the softmax never waits (13% faster than S of whole tiles).
// Why blocks: the hot code of the warps together has to stay in the instruction cache.  With a row
// of 128 scores unrolled it was about 26 KB, and a tile's softmax took 1.7 times as long as in a
// kernel of its own.
template <int D>
struct TcShape {
  static constexpr int kTile = 128;                          // slots per K/V tile
  static constexpr int kChunks = kTile / kChunkSlots;        // 16-slot TMA chunks per tile
  static constexpr int kBlock = 64;                          // slots per softmax block
  static constexpr int kBlockChunks = kBlock / kChunkSlots;
  static constexpr bool kTileS = D == 128;                   // S by tiles; else by blocks, two ahead
  static constexpr int kSSlots = kTileS ? kTile : kBlock;    // slots (N) of an S product
  static constexpr int kHalves = D / 64;                     // 64-column halves of a row
  // A K (or V) tile, a ring stage: 8-row groups, each its 64-column halves one after the other
  // (8 rows of 128 bytes in the 128-byte swizzle), so that a 16-slot chunk is one TMA box.
  static constexpr int kGroupBytes = kHalves * 1024;
  static constexpr int kChunkBytes = 2 * kGroupBytes;
  static constexpr int kKVBytes = kChunks * kChunkBytes;
  static constexpr int kStages = D == 128 ? 5 : 10;          // K and V tiles in flight
  static constexpr int kQHalfBytes = 128 * 128;              // one half of a Q tile
  static constexpr int kQBytes = kHalves * kQHalfBytes;
  static constexpr int kOffRing = 2 * kQBytes;               // Q tiles at 0
  static constexpr int kOffBar = kOffRing + kStages * kKVBytes;
  // full, empty [kStages]; q_full, q_empty, o_full, pv_done [2]; s_full, p_full [2][2];
  // item_full, item_empty [kItems]; mma_done; turn [2]
  static constexpr int kItems = 4;                           // items handed out ahead
  static constexpr int kBars = 2 * kStages + 19 + 2 * kItems;
  static constexpr int kOffItems = kOffBar + (kBars * 8 + 15) / 16 * 16;
  static constexpr int kOffMisc = kOffItems + kItems * (int)sizeof(PrefillItem);
  static constexpr int kSmem = 1024 + kOffMisc + 16;
  static constexpr uint32_t kTmemCols = 512;
  static constexpr int kOffO = 2 * kTile;                    // TMEM column of O_0 (S_0 at 0)
  // softmax: warps 0-3 (Q tile 0) and 4-7 (Q tile 1); TMA producers of K (8) and of Q and V (9,
  // which also fetches the items); the MMA issuers of Q tile 0 (10) and 1 (11).
  static constexpr int kProducerWarp = 8, kVProducerWarp = 9, kMmaWarp = 10;
  static constexpr int kThreads = 12 * 32;
  static_assert(D == 64 || D == 128, "head_dim 64 or 128");
  static_assert(kOffO + 2 * D <= (int)kTmemCols, "TMEM columns");
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

// Scores of the slots past `seen` (of a block's 64) become -inf: the causal edge, the chunk's end.
__device__ __forceinline__ void mask_scores(uint32_t (&r)[2][32], int seen) {
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int c = 0; c < 32; ++c)
      if (32 * x + c > seen) r[x][c] = 0xFF800000u;
}
__device__ __forceinline__ float max_score(const uint32_t (&r)[2][32]) {
  float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
  for (int c = 0; c < 32; c += 4)
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      m[2 * x] = fmaxf(fmaxf(m[2 * x], __uint_as_float(r[x][c])), __uint_as_float(r[x][c + 1]));
      m[2 * x + 1] = fmaxf(fmaxf(m[2 * x + 1], __uint_as_float(r[x][c + 2])), __uint_as_float(r[x][c + 3]));
    }
  return fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
}

template <typename OutT>
__device__ __forceinline__ void store_row32(OutT *dst, const uint32_t (&o)[32], float scale) {
  if constexpr (std::is_same<OutT, float>::value) {
#pragma unroll
    for (int e = 0; e < 32; e += 4)
      *reinterpret_cast<float4 *>(dst + e) =
          make_float4(__uint_as_float(o[e]) * scale, __uint_as_float(o[e + 1]) * scale,
                      __uint_as_float(o[e + 2]) * scale, __uint_as_float(o[e + 3]) * scale);
  } else {
#pragma unroll
    for (int e = 0; e < 32; e += 8)
      *reinterpret_cast<uint4 *>(dst + e) = make_uint4(
          pack_bf16x2(__uint_as_float(o[e]) * scale, __uint_as_float(o[e + 1]) * scale),
          pack_bf16x2(__uint_as_float(o[e + 2]) * scale, __uint_as_float(o[e + 3]) * scale),
          pack_bf16x2(__uint_as_float(o[e + 4]) * scale, __uint_as_float(o[e + 5]) * scale),
          pack_bf16x2(__uint_as_float(o[e + 6]) * scale, __uint_as_float(o[e + 7]) * scale));
  }
}

// Items of a launch: every (KV head, query block, split), KV head fastest, the query blocks in the
// plan's order.  False: the sequence was refused, or has fewer splits.
__device__ __forceinline__ bool decode_item(const PrefillView &v, int id, int nblocks, int tile,
                                            PrefillItem &it) {
  const int Hkv = v.n_kv_heads, R = 128 / (v.n_q_heads / Hkv);
  const int rest = id / Hkv, z = rest / nblocks;
  const int2 blk = v.order[rest - z * nblocks];  // (sequence, query block of its chunk)
  const int4 si = v.seq_info[blk.x];
  const int L = si.x, n = si.y, qb0 = blk.y * 2 * R;
  const int zs = prefill_splits(L, v.splits);
  if (L < 0 || z >= zs) return false;
  // Split z of the sequence's zs takes tiles t0 .. t1 - 1: the cached part's whole tiles cut
  // evenly, the last split also the rest (the chunk's own slots, the causal edge).  Every split
  // starts at or before slot L - tile, which every row attends, so no row of a split is empty.
  const int rows_q0 = min(R, n - qb0), rows_q1 = max(0, min(R, n - qb0 - R));
  const int end0 = L + qb0 + rows_q0, end1 = rows_q1 > 0 ? end0 + rows_q1 : 0;
  const int n0 = (end0 + tile - 1) / tile, n1 = (end1 + tile - 1) / tile;
  const int ntiles = max(n0, n1), Lt = L / tile;  // (Lt * zs: below 2^31 / 128 * 32)
  const int t0 = z * Lt / zs, t1 = z + 1 == zs ? ntiles : (z + 1) * Lt / zs;
  it.valid = 1;
  it.b = blk.x;
  it.g = id - rest * Hkv;
  it.L = L;
  it.n = n;
  it.qb0 = qb0;
  it.row0 = si.z;
  it.z = z;
  it.zs = zs;
  it.t0 = t0;
  it.nt0 = max(0, min(t1, n0) - t0);
  it.nt1 = max(0, min(t1, n1) - t0);
  it.end0 = end0;
  it.end1 = end1;
  return true;
}

// One CTA per SM (shared memory and 512 TMEM columns).
template <int D, typename OutT>
__global__ void __launch_bounds__(TcShape<D>::kThreads, 1)
    prefill_attn_kernel(const __grid_constant__ CUtensorMap tmap_q,
                        const __grid_constant__ CUtensorMap tmap_k,
                        const __grid_constant__ CUtensorMap tmap_v, const PrefillView v) {
  using S = TcShape<D>;
  const int Hq = v.n_q_heads, Hkv = v.n_kv_heads, G = Hq / Hkv, R = 128 / G;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + S::kOffBar);
  uint64_t *empty = full + S::kStages, *q_full = empty + S::kStages, *q_empty = q_full + 2;
  uint64_t *o_full = q_full + 4, *pv_done = q_full + 6, *s_full = q_full + 8, *p_full = q_full + 12;
  uint64_t *item_full = q_full + 16, *item_empty = item_full + S::kItems;
  uint64_t *mma_done = item_empty + S::kItems, *turn = mma_done + 1;
  PrefillItem *items = reinterpret_cast<PrefillItem *>(smem + S::kOffItems);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + S::kOffMisc);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  const int tid = threadIdx.x, warp = __shfl_sync(kFull, tid >> 5, 0), lane = tid & 31;
  if (tid == 0) {
    // a stage is free once the products of both Q tiles that read it completed
    for (int s = 0; s < S::kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 2);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&q_full[q], 1);
      mbar_init(&q_empty[q], 1);
      mbar_init(&o_full[q], 1);
      mbar_init(&pv_done[q], 1);
      for (int x = 2 * q; x < 2 * q + 2; ++x) {
        mbar_init(&s_full[x], 1);
        mbar_init(&p_full[x], 4);  // the softmax group has written a block's P (one arrival per warp)
      }
    }
    for (int x = 0; x < S::kItems; ++x) {
      mbar_init(&item_full[x], 1);
      mbar_init(&item_empty[x], 11);     // 8 softmax warps, the K producer, 2 MMA warps
    }
    mbar_init(mma_done, 2);
    mbar_init(&turn[0], 4);  // the turn of Q tile 0's / 1's softmax group (one arrival per warp)
    mbar_init(&turn[1], 4);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == S::kProducerWarp && lane == 0) {
    prefetch_tensormap(&tmap_q);
    prefetch_tensormap(&tmap_k);
    prefetch_tensormap(&tmap_v);
  }
  if (warp == S::kMmaWarp) tmem_alloc<S::kTmemCols>(tmem_slot);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_dependency_wait();  // the plan, the rotated queries and the stored rows
  grid_launch_dependents();
  if (blockIdx.x == 0 && warp < S::kProducerWarp) {  // the slot counters (the plan's blocks read them all)
    for (int b = tid; b < v.batch; b += S::kProducerWarp * 32) {
      const int4 si = v.seq_info[b];
      if (si.x >= 0) v.num_slots[b] = si.x + si.y;
    }
  }
  // ring and data waits: the launch's limit; item hand-over and the draining of in-flight work
  // keep the default 2 s
  const uint64_t wait_lim = data_wait_limit(v.wait_ns);
  // The next item: every role reads it from the item ring and frees the entry.
  auto give_up = [&]() {
    if (lane == 0 && !*abort_flag) {
      record_error(v.err, HAM_DEVERR_TIMEOUT);
      *abort_flag = 1;
    }
  };
  auto next_item = [&](uint32_t k, PrefillItem &it) -> bool {
    const uint32_t x = k % S::kItems;
    if (!warp_wait_small(&item_full[x], (k / S::kItems) & 1u, abort_flag, kWaitLimitNs)) {
      give_up();
      return false;
    }
    it = items[x];
    __syncwarp();
    if (lane == 0) mbar_arrive(&item_empty[x]);
    return uniform(it.valid) != 0;
  };
  uint32_t issued = 0, q_issued[2] = {0u, 0u};  // producers: ring entries past the last one; Q loads

  if (warp >= S::kProducerWarp) {
    if (warp < S::kMmaWarp) {
      // ---------------------------------------------------------- producers: TMA copies
      // One warp streams the K tiles, the other Q and the V tiles, into one ring in the order
      // K_0 V_0 K_1 V_1 ... (the order the products read them).  A chunk at or past the item's
      // end is not copied: its rows are never read (whole chunks) or zeroed (V, the last one).
      const bool is_v = warp == S::kVProducerWarp;
      const CUtensorMap *map = is_v ? &tmap_v : &tmap_k;
      const uint64_t pol_first = policy_evict_first(), pol_last = policy_evict_last();
      uint32_t e = is_v ? 1 : 0;  // ring entry of the next tile
      bool ok = true;
      PrefillItem it;
      // The V producer hands the items out: the next one once it has issued this one's last copies
      // (earlier would give a CTA two of the launch's last items while others have none).
      const int nblocks = v.next_item[1];
      const int total = Hkv * nblocks * v.splits;
      auto fetch = [&](uint32_t k) -> bool {
        const uint32_t x = k % S::kItems;
        if (k >= S::kItems && !warp_wait_small(&item_empty[x], ((k / S::kItems) - 1) & 1u,
                                               abort_flag, kWaitLimitNs)) {
          give_up();
          return false;
        }
        it = PrefillItem{};
        for (;;) {
          int id = 0;
          if (lane == 0) id = atomicAdd(v.next_item, 1);
          id = uniform(id);
          if (id >= total || decode_item(v, id, nblocks, S::kTile, it)) break;
        }
        if (lane == 0) {
          items[x] = it;
          mbar_arrive(&item_full[x]);
        }
        return uniform(it.valid) != 0;
      };
      for (uint32_t k = 0; ok; ++k) {
        if (is_v ? !fetch(k) : !next_item(k, it)) break;
        const int nts = uniform(max(it.nt0, it.nt1)), kv_end = uniform(max(it.end0, it.end1));
        // a sequence with several query blocks re-reads its K/V from L2
        const uint64_t pol_kv = it.n > 2 * R ? pol_last : pol_first;
        if (is_v) {  // Q (so that the K tiles do not wait for the previous item's last product)
          const int nq = it.nt1 > 0 ? 2 : 1;
          for (int q = 0; ok && q < nq; ++q) {
            if (q_issued[q] > 0 &&
                !warp_wait_small(&q_empty[q], (q_issued[q] - 1) & 1u, abort_flag, wait_lim)) {
              give_up();
              ok = false;
              break;
            }
            ++q_issued[q];
            if (elect_one()) {
              mbar_arrive_tx(&q_full[q], (uint32_t)S::kQBytes);
              tma_load_4d(smem + q * S::kQBytes, &tmap_q, 0, it.g * G, it.row0 + it.qb0 + q * R, 0,
                          &q_full[q], pol_first);
            }
            __syncwarp();
          }
          if (!ok) break;
        }
        // Page-table entries of 32 chunks (4 tiles) at a time, one per lane, requested a batch
        // ahead: lane l holds the pool row of chunk base + l (-1: at or past the item's end; -2:
        // a page outside the pool).
        const int nchunks = (kv_end + kChunkSlots - 1) / kChunkSlots;
        auto lookup = [&](int base) {
          int row = -1;
          if (base + lane < nchunks) {
            const int slot0 = (base + lane) * kChunkSlots;
            const int page = v.page_table[(int64_t)it.b * v.max_pages + slot0 / v.page_slots];
            row = page < 0 || page >= v.pool_pages
                      ? -2
                      : (int)(((int64_t)page * Hkv + it.g) * v.page_slots + slot0 % v.page_slots);
          }
          return row;
        };
        constexpr int kTilesPerBatch = 32 / S::kChunks;
        const int cbase = it.t0 * S::kChunks;  // the item's first chunk
        int row = lookup(cbase), row_next = lookup(cbase + 32);
        for (int i = 0; i < nts; ++i, e += 2) {
          if (i > 0 && i % kTilesPerBatch == 0) {
            row = row_next;
            row_next = lookup(cbase + (i / kTilesPerBatch + 1) * 32);
          }
          if (__any_sync(kFull, row == -2)) {  // the plan validated the table: ends the CTA
            if (lane == 0) {
              record_error(v.err, HAM_DEVERR_PAGE);
              *abort_flag = 1;
            }
            ok = false;
            break;
          }
          const uint32_t st = e % S::kStages;
          if (e >= S::kStages && !warp_wait_small(&empty[st], ((e / S::kStages) - 1) & 1u,
                                                 abort_flag, wait_lim)) {
            give_up();
            ok = false;
            break;
          }
          const int nck = min(S::kChunks, nchunks - cbase - i * S::kChunks);
          const int at = (i % kTilesPerBatch) * S::kChunks;
          if (elect_one()) mbar_arrive_tx(&full[st], (uint32_t)(nck * kChunkSlots * D * 2));
          uint8_t *dst = smem + S::kOffRing + st * S::kKVBytes;
#pragma unroll 1
          for (int c = 0; c < nck; ++c) {
            const int r = __shfl_sync(kFull, row, at + c);
            if (elect_one()) tma_load_4d(dst + c * S::kChunkBytes, map, 0, 0, 0, r >> 3, &full[st], pol_kv);
          }
        }
      }
      issued = e;
    } else {
      // ---------------------------------------------------------- MMA issue (one thread a Q tile)
      // The first S of an item (two where S goes by blocks), then block by block O += P V once the
      // softmax group has written P, and the S whose columns are free then.  What holds an item's
      // end takes only the 16-slot chunks it reaches (N of S, K of P V).  Both warps release every
      // K and V stage by a commit, also where their Q tile has no product: commits complete in the
      // order of issue, so a warp releases the ring's stages in their order (but for a tile's V and the
      // next tile's K, which change places).  The producers need that: a stage of an odd ring is
      // filled by the two in turn, and a producer that waits, by parity, for the other's fill to be
      // released relies on the fill before that one having been released too, which follows from the
      // release its own last entry waited for, five entries earlier.  Everything the products'
      // operands depend on is kept uniform over the warp: with per-thread values an issue took
      // about 100 cycles, against the 32 to 64 that the product itself takes.
      constexpr uint32_t id_o = idesc_bf16(128, D, true);  // P from TMEM, MN-major V
      const int q = warp - S::kMmaWarp;
      const uint32_t ring = smem_u32(smem + S::kOffRing);
      const uint64_t q_desc = smem_desc_sw128(smem_u32(smem) + q * S::kQBytes, 16, 1024);
      const uint32_t d_s = tmem + q * S::kTile, d_o = tmem + S::kOffO + q * D;
      uint32_t e = 0, pc = 0, qc = 0;  // ring entry of the item's first K tile; parities of P; Q loads
      bool ok = true;
      PrefillItem it;
      for (uint32_t k = 0; ok && next_item(k, it); ++k) {
        const int nt = uniform(q ? it.nt1 : it.nt0), nts = uniform(max(it.nt0, it.nt1));
        const int base = uniform(it.t0) * S::kTile, end = uniform(q ? it.end1 : it.end0) - base;
        const int kv_end = uniform(max(it.end0, it.end1)) - base;  // (from the item's first slot)
        // blocks of this Q tile (a tile without rows has no end)
        const int nb = nt == 0 ? 0 : min(2 * nt, (end + S::kBlock - 1) / S::kBlock);
        const uint32_t e0 = e;
        e += 2 * nts;
        auto chunks = [&](int from, int most) {  // 16-slot chunks that this Q tile reaches
          return min(most, (end - from + kChunkSlots - 1) / kChunkSlots);
        };
        auto wait_entry = [&](uint32_t x) {
          return warp_wait_small(&full[x % S::kStages], (x / S::kStages) & 1u, abort_flag, wait_lim);
        };
        // S of tile t / 2 or of block t, and the release of K and Q after their last.
        auto issue_s = [&](int t) {
          const uint32_t st = (e0 + 2 * (t >> 1)) % S::kStages, buf = S::kTileS ? 0 : t & 1;
          const uint64_t b0 = smem_desc_sw128(
              ring + st * S::kKVBytes + buf * (S::kBlock / 8) * S::kGroupBytes, 16, S::kGroupBytes);
          const uint32_t id_s = idesc_bf16(
              128, kChunkSlots * chunks(t * S::kBlock, S::kSSlots / kChunkSlots), false);  // K-major
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk)
            tc_mma(d_s + buf * S::kBlock,
                   q_desc + (uint64_t)(((kk >> 2) * S::kQHalfBytes + (kk & 3) * 32) >> 4),
                   b0 + (uint64_t)(((kk >> 2) * 1024 + (kk & 3) * 32) >> 4), id_s, kk > 0);
          tc_commit(&s_full[2 * q + buf]);
          const bool last = t + (S::kTileS ? 2 : 1) >= nb;
          if (S::kTileS || buf == 1 || last) tc_commit(&empty[st]);
          if (last) tc_commit(&q_empty[q]);
        };
        if (nb > 0) {
          ok = warp_wait_small(&q_full[q], qc & 1u, abort_flag, wait_lim);
          if (!ok) break;
          ok = wait_entry(e0);
          if (!ok) break;
          ++qc;
          tc_fence_after();
          if (elect_one()) issue_s(0);
          __syncwarp();
          if (!S::kTileS && nb > 1 && elect_one()) issue_s(1);
          __syncwarp();
        }
        for (int t = 0; t < nb; ++t) {
          const uint32_t buf = t & 1, ev = e0 + 2 * (t >> 1) + 1, sv = ev % S::kStages;  // V's entry
          if (buf == 0) {  // a new tile: its values, and the keys of the next one
            ok = wait_entry(ev);
            if (!ok) break;
            if ((t >> 1) + 1 < nt) {
              ok = wait_entry(ev + 1);
              if (!ok) break;
            }
            const int z0 = kv_end - t * S::kBlock;  // rows of the tile >= z0 are past the last slot
            if (z0 < S::kTile && (z0 & (kChunkSlots - 1))) {
              // slots past the end get p = 0; zero their value rows (to the end of the last chunk
              // the products read) so that stale bits never reach O (both warps may do it)
              uint8_t *vt = smem + S::kOffRing + sv * S::kKVBytes;
              const int pieces = (kChunkSlots - (z0 & (kChunkSlots - 1))) * S::kHalves * 8;
              for (int x = lane; x < pieces; x += 32) {  // 16-byte pieces of rows z0 ..
                const int row = z0 + x / (S::kHalves * 8), y = x % (S::kHalves * 8);
                *reinterpret_cast<uint4 *>(vt + (row >> 3) * S::kGroupBytes + (y >> 3) * 1024 +
                                           (row & 7) * 128 + (y & 7) * 16) = make_uint4(0u, 0u, 0u, 0u);
              }
              fence_proxy_async_smem();
              __syncwarp();
            }
          }
          ok = warp_wait_small(&p_full[2 * q + buf], (pc >> buf) & 1u, abort_flag, wait_lim);
          if (!ok) break;
          pc ^= 1u << buf;
          tc_fence_after();
          const int nc = chunks(t * S::kBlock, S::kBlockChunks);
          const uint32_t a0 = d_s + buf * S::kBlock;
          const uint64_t v0 = smem_desc_sw128(  // MN-major: halves 1024 bytes apart
              ring + sv * S::kKVBytes + buf * (S::kBlockChunks * S::kChunkBytes), 1024, S::kGroupBytes);
          if (elect_one()) {
#pragma unroll
            for (int c = 0; c < S::kBlockChunks; ++c)
              if (c < nc)
                tc_mma_tmem_a(d_o, a0 + c * 8, v0 + (uint64_t)(c * S::kChunkBytes >> 4), id_o,
                              t > 0 || c > 0);
            tc_commit(&pv_done[q]);
            if (t + 1 == nb) tc_commit(&o_full[q]);
            if (S::kTileS) {
              if (buf == 1 && t + 1 < nb) issue_s(t + 1);
            } else if (t + 2 < nb) {
              issue_s(t + 2);
            }
            if (buf == 1 || t + 1 == nb) tc_commit(&empty[sv]);
          }
          __syncwarp();
        }
        for (uint32_t x = e0 + 2 * nt; ok && x != e; ++x) {  // tiles it does not reach
          ok = wait_entry(x);
          if (ok && elect_one()) tc_commit(&empty[x % S::kStages]);
          __syncwarp();
        }
      }
      if (!ok) give_up();
      // every MMA issued completes before the tensor memory is freed
      if (elect_one()) {
        tc_commit(mma_done);
        thread_wait(mma_done, 0u, abort_flag, false);
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------ softmax groups
    // Thread = TMEM lane = row m of Q tile q.  Each row's scores arrive whole in its own thread,
    // so the row maximum and sum need no shuffles.
    const int q = warp >> 2, m = tid & 127;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t t_s = tmem + lane_base + q * S::kTile;  // the two blocks of S_q, then P_q
    const uint32_t t_o = tmem + lane_base + S::kOffO + q * D;
    const float sl2 = (float)(1.4426950408889634 / sqrt((double)D));  // 1/sqrt(d), log2(e)
    // phase parities of s_full; blocks, items and turns so far
    uint32_t sp = 0, np = 0, oc = 0, turns = turns_before(q);
    bool ok = true;
    for (uint32_t k = 0;; ++k) {
      int tbase, tend, lim, lim_min;  // first slot of the block, of the item's end; row limits
      int turn_end;                   // the blocks before this slot belong to tiles that take turns
      int64_t orow = -1;              // the row's place in out (or in the split's partials)
      bool whole;
      {
        PrefillItem it;
        if (!next_item(k, it)) break;
        const int nt = q ? it.nt1 : it.nt0;
        if (nt == 0) continue;
        const int j = it.qb0 + q * R + m / G;  // the row's index in the sequence's chunk
        lim = it.L + min(j, it.n - 1);         // last slot it attends (rows past n: not stored)
        lim_min = it.L + it.qb0 + q * R;       // smallest limit of the tile's stored rows
        tbase = it.t0 * S::kTile;
        tend = min(tbase + nt * S::kTile, q ? it.end1 : it.end0);
        whole = it.zs == 1;
        // Q tile 1's softmax of a tile that both read follows Q tile 0's, which follows Q tile 1's of
        // the shared tile before, in this item or an earlier one.
        turn_end = tbase + turn_tiles(it.nt0, it.nt1) * S::kTile;
        if (j < it.n)
          orow = ((whole ? 0 : (int64_t)it.z * v.rows) + it.row0 + j) * Hq + it.g * G + m % G;
      }
      float m_run = -INFINITY, l_run = 0.f;
      for (uint32_t buf = 0; tbase < tend; tbase += S::kBlock, buf ^= 1u, ++np) {
        if (!S::kTileS || buf == 0) {  // new scores
          if (!warp_wait_small(&s_full[2 * q + buf], (sp >> buf) & 1u, abort_flag, wait_lim)) {
            ok = false;
            break;
          }
          sp ^= 1u << buf;
          if (S::kTileS && tbase < turn_end) {
            if (!warp_wait_small(&turn[q], turns & 1u, abort_flag, wait_lim)) {
              ok = false;
              break;
            }
            ++turns;
          }
          tc_fence_after();
        }
        const uint32_t t_b = t_s + buf * S::kBlock;
        uint32_t r[2][32];
        tmem_ld32(t_b, r[0]);
        tmem_ld32(t_b + 32, r[1]);
        tmem_wait_ld();
        if (tbase + S::kBlock - 1 > lim_min) mask_scores(r, lim - tbase);
        // Running maximum in the exp2 domain, raised lazily: only when a score passes it by more
        // than kRescaleSlack (p then stays below 2^kRescaleSlack), so O is rarely rescaled.  The
        // item's first block always raises it (its first slot is attended by every row).
        const float mx = max_score(r) * sl2;
        const bool raise = mx > m_run + kRescaleSlack;
        if (__any_sync(kFull, raise)) {
          const float alpha = raise ? ex2(m_run - mx) : 1.f;
          if (__any_sync(kFull, raise && m_run != -INFINITY)) {  // (the first block overwrites O)
            // once O holds the previous block too (the phase before this block's)
            if (!warp_wait_small(&pv_done[q], (np - 1) & 1u, abort_flag, wait_lim)) {
              ok = false;
              break;
            }
            tc_fence_after();
#pragma unroll 1
            for (int c0 = 0; c0 < D; c0 += 32) {
              uint32_t o[32];
              tmem_ld32(t_o + c0, o);
              tmem_wait_ld();
#pragma unroll
              for (int x = 0; x < 32; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * alpha);
              tmem_st32(t_o + c0, o);
            }
          }
          if (raise) m_run = mx;
          l_run *= alpha;
        }
        // P in two parts, the first stored while the second is formed (in one part: 8% slower)
        float rs0 = 0.f, rs1 = 0.f, rs2 = 0.f, rs3 = 0.f;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          uint32_t pk[16];
#pragma unroll
          for (int c = 0; c < 32; c += 4) {
            const float p0 = ex2(fmaf(__uint_as_float(r[x][c]), sl2, -m_run));
            const float p1 = ex2(fmaf(__uint_as_float(r[x][c + 1]), sl2, -m_run));
            const float p2 = ex2(fmaf(__uint_as_float(r[x][c + 2]), sl2, -m_run));
            const float p3 = ex2(fmaf(__uint_as_float(r[x][c + 3]), sl2, -m_run));
            rs0 += p0;
            rs1 += p1;
            rs2 += p2;
            rs3 += p3;
            pk[c / 2] = pack_bf16x2(p0, p1);
            pk[c / 2 + 1] = pack_bf16x2(p2, p3);
          }
          if (x == 1 && S::kTileS && tbase < turn_end && (buf == 1 || tbase + S::kBlock >= tend) &&
              lane == 0)
            mbar_arrive(&turn[q ^ 1]);
          tmem_st16(t_b + 16 * x, pk);  // 32 probabilities as 16 bf16 pairs
        }
        l_run += (rs0 + rs1) + (rs2 + rs3);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[2 * q + buf]);
      }
      if (!ok || !warp_wait_small(&o_full[q], oc & 1u, abort_flag, wait_lim)) {
        ok = false;
        break;
      }
      ++oc;
      tc_fence_after();
      if (whole) {  // normalised output
        const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
        OutT *dst = static_cast<OutT *>(v.out) + orow * D;
#pragma unroll 1
        for (int c0 = 0; c0 < D; c0 += 32) {
          uint32_t o[32];
          tmem_ld32(t_o + c0, o);
          tmem_wait_ld();
          if (orow >= 0) store_row32<OutT>(dst + c0, o, inv);
        }
      } else {  // this split's partial: O in units of 2^m_run, the running max and sum
        float *dst = v.part_o + orow * D;
#pragma unroll 1
        for (int c0 = 0; c0 < D; c0 += 32) {
          uint32_t o[32];
          tmem_ld32(t_o + c0, o);
          tmem_wait_ld();
          if (orow >= 0) store_row32<float>(dst + c0, o, 1.f);
        }
        if (orow >= 0) v.part_ml[orow] = make_float2(m_run, l_run);
      }
    }
    if (!ok) give_up();
  }
  // all tensor-memory reads and MMAs are done: free the columns
  volatile uint32_t *issued_s = reinterpret_cast<volatile uint32_t *>(items);  // K, V, Q tiles
  tc_fence_before();
  __syncthreads();
  if (lane == 0 && warp == S::kProducerWarp) issued_s[0] = issued;
  if (lane == 0 && warp == S::kVProducerWarp) {
    issued_s[1] = issued;
    issued_s[2] = q_issued[0];
    issued_s[3] = q_issued[1];
  }
  if (warp == S::kMmaWarp) {
    tc_fence_after();
    tmem_dealloc<S::kTmemCols>(tmem);
  }
  __syncthreads();
  if (tid == 0 && *abort_flag) {
    // after an abort, every copy this CTA issued lands before the CTA can exit (without one, the
    // MMA warp waited for every copy): the entries whose ring stage was not filled again
    for (uint32_t w = 0; w < 2; ++w)
      for (uint32_t x = w; x < issued_s[w]; x += 2) {
        const uint32_t y = x + S::kStages;  // the entry that would reuse the stage
        if (y >= issued_s[y & 1]) thread_wait(&full[x % S::kStages], (x / S::kStages) & 1u, abort_flag, false);
      }
    for (int q = 0; q < 2; ++q)
      if (issued_s[2 + q] > 0) thread_wait(&q_full[q], (issued_s[2 + q] - 1) & 1u, abort_flag, false);
  }
}

// ------------------------------------------------------------------------------------
// 4. merge of the split partials (only when the attention grid has splits)
// ------------------------------------------------------------------------------------
// out = sum_z 2^(m_z - M) O_z / sum_z 2^(m_z - M) l_z over the splits z of the row's sequence, in
// split order (M = max_z m_z; the split-softmax merge of the decode combine).  One warp per
// (row, head), D / 32 elements a lane; rows of sequences that were not split (written by the
// attention itself) or that the plan refused are left alone.  Lane z takes split z's (max, sum) and
// weight, and the partials are read kMergeBatch at a time: the kernel is bound by its round trips
// to L2 (one split after the other took 18 us for 2,048 rows of 19 splits).
constexpr int kMergeWarps = 8, kMergeBatch = 8;
static_assert(kPrefillMaxSplits <= 32, "one lane a split");
template <int D, typename OutT>
__global__ void __launch_bounds__(kMergeWarps * 32) prefill_merge_kernel(const PrefillView v) {
  constexpr int kPer = D / 32;  // elements a lane
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Hq = v.n_q_heads;
  const int64_t rh = (int64_t)blockIdx.x * kMergeWarps + warp;  // (row, head)
  grid_dependency_wait();
  if (rh >= (int64_t)v.rows * Hq) return;
  const int r = (int)(rh / Hq);
  int lo = 0, hi = v.batch - 1;  // the row's sequence: the last b with offsets[b] <= r
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (v.offsets[mid] <= r) lo = mid; else hi = mid - 1;
  }
  const int4 si = v.seq_info[lo];
  if (si.x < 0) return;
  const int zs = prefill_splits(si.x, v.splits);
  if (zs <= 1) return;
  const int64_t zstride = (int64_t)v.rows * Hq;
  const float2 ml = lane < zs ? v.part_ml[lane * zstride + rh] : make_float2(-INFINITY, 0.f);
  const float M = warp_max_f32(ml.x);
  const float w = ml.x == -INFINITY ? 0.f : ex2(ml.x - M);
  float num[kPer], den = 0.f;
#pragma unroll
  for (int e = 0; e < kPer; ++e) num[e] = 0.f;
  const float *po = v.part_o + rh * D + lane * kPer;
  for (int z0 = 0; z0 < zs; z0 += kMergeBatch) {
    float o[kMergeBatch][kPer];
#pragma unroll
    for (int x = 0; x < kMergeBatch; ++x) {
      const float *src = po + (int64_t)min(z0 + x, zs - 1) * zstride * D;
      if constexpr (kPer == 4) {
        const float4 y = *reinterpret_cast<const float4 *>(src);
        o[x][0] = y.x; o[x][1] = y.y; o[x][2] = y.z; o[x][3] = y.w;
      } else {
        const float2 y = *reinterpret_cast<const float2 *>(src);
        o[x][0] = y.x; o[x][1] = y.y;
      }
    }
#pragma unroll
    for (int x = 0; x < kMergeBatch; ++x) {
      const int z = z0 + x;
      const float wz = __shfl_sync(kFull, w, z & 31), lz = __shfl_sync(kFull, ml.y, z & 31);
      if (z < zs) {
        den += wz * lz;
#pragma unroll
        for (int e = 0; e < kPer; ++e) num[e] += wz * o[x][e];
      }
    }
  }
  const float inv = den > 0.f ? 1.f / den : 0.f;
  OutT *dst = static_cast<OutT *>(v.out) + rh * D + lane * kPer;
#pragma unroll
  for (int e = 0; e < kPer; ++e) {
    if constexpr (std::is_same<OutT, float>::value)
      dst[e] = num[e] * inv;
    else
      dst[e] = __float2bfloat16_rn(num[e] * inv);
  }
}

// A launch with programmatic dependent launch: the kernel may start before its predecessor on the
// stream ends and waits for it (griddepcontrol.wait) before it reads or writes anything that the
// predecessor writes or reads.
template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*kernel)(KArgs...), unsigned grid, int threads, size_t smem,
                             cudaStream_t stream, const Args &...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int D, typename OutT>
cudaError_t launch_attn(const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv,
                        const PrefillView &v, cudaStream_t stream) {
  using S = TcShape<D>;
  cudaError_t e = cudaFuncSetAttribute(prefill_attn_kernel<D, OutT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, S::kSmem);
  if (e != cudaSuccess) return e;
  const int64_t items = (int64_t)v.n_kv_heads * v.blocks * v.splits;
  const unsigned grid = (unsigned)(items < v.sms ? items : v.sms);  // persistent: one CTA an SM
  e = launch_dependent(prefill_attn_kernel<D, OutT>, grid, S::kThreads, S::kSmem, stream, tq, tk,
                       tv, v);
  if (e != cudaSuccess || v.splits == 1) return e;
  const int64_t pairs = (int64_t)v.rows * v.n_q_heads;
  return launch_dependent(prefill_merge_kernel<D, OutT>,
                          (unsigned)((pairs + kMergeWarps - 1) / kMergeWarps), kMergeWarps * 32, 0,
                          stream, v);
}

template <typename OutT>
cudaError_t launch_all(const CUtensorMap &tk, const CUtensorMap &tv, const PrefillView &v,
                       cudaStream_t stream) {
  const int G = v.n_q_heads / v.n_kv_heads;
  CUtensorMap tq;  // the chunk's queries, rotated in place by the RoPE kernel
  if (make_rows_tensor_map(&tq, v.q, v.rows, v.n_q_heads, v.head_dim, G, 128 / G) != 0)
    return cudaErrorInvalidValue;
  int qb_shift = 0;  // (a power of two)
  while (1 << qb_shift < prefill_query_rows(G)) ++qb_shift;
  prefill_plan_kernel<<<(unsigned)v.batch, kPlanThreads, 0, stream>>>(v, qb_shift);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // RoPE: a thread for every eight pairs of the row's heads, in equal passes of at most kRopeThreads
  const int octs = (v.n_q_heads + v.n_kv_heads) * (v.head_dim / 16);
  const int passes = (octs + kRopeThreads - 1) / kRopeThreads;
  const int threads = max(64, ((octs + passes - 1) / passes + 31) / 32 * 32);
  const auto rope = v.head_dim == 128
                        ? (passes > 1 ? prefill_rope_kernel<128, OutT, true> : prefill_rope_kernel<128, OutT, false>)
                        : (passes > 1 ? prefill_rope_kernel<64, OutT, true> : prefill_rope_kernel<64, OutT, false>);
  e = launch_dependent(rope, (unsigned)v.rows, threads, 0, stream, v);
  if (e != cudaSuccess) return e;
  return v.head_dim == 128 ? launch_attn<128, OutT>(tq, tk, tv, v, stream)
                           : launch_attn<64, OutT>(tq, tk, tv, v, stream);
}

}  // namespace

bool prefill_supported(int head_dim, int group) {
  return (head_dim == 64 || head_dim == 128) &&
         (group == 1 || group == 2 || group == 4 || group == 8);
}

// Two Q tiles of 128 (row, head) pairs per CTA.
int prefill_query_rows(int group) { return 256 / group; }

cudaError_t launch_prefill(const CUtensorMap &tk, const CUtensorMap &tv, const PrefillView &v,
                           int out_dtype, cudaStream_t stream) {
  return out_dtype == HAM_DTYPE_F32 ? launch_all<float>(tk, tv, v, stream)
                                    : launch_all<__nv_bfloat16>(tk, tv, v, stream);
}

}  // namespace ham
