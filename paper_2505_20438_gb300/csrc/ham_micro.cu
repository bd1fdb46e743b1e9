// Micro-step attention: one step of a decoder whose per-sequence cache is a handful of slots.
//
// HAMburger's micro-step decoder (Sec. 3.3; Sec. 4.1: four layers with the base model's
// configuration) generates the tokens of a macro-step one by one, conditioned on hidden states
// of several middle layers of the base model as context.  Its attention reads only that local
// context and the micro-tokens produced so far, never the base model's cache, so its cost does
// not grow with the sequence (Sec. 3.7, the constant c of the speed-up model).  Per layer and
// micro-step the work is: rotate q and k at the new entry's position, append k and v, attend
// over at most 16 entries.  The general decode step (plan, split, combine: two launches) is
// built for caches of thousands of slots; here one kernel does everything:
//  - one CTA per (sequence, KV head); the CTAs of a sequence form a thread-block cluster, whose
//    barrier orders every CTA's read of the slot counter before rank 0 advances it (CTAs arrive as
//    soon as they have read it and wait only at their end);
//  - the step is a chain of latencies, so what does not depend on the caller's inputs (the counters,
//    the page entry, then the old entries and the cos/sin at the position) is read before the
//    programmatic-dependency wait when the host allows it (`early`: the launch before wrote another
//    layer), beside the end of the previous kernel; the query heads, the new key and value and the
//    token count follow the wait in one round trip;
//  - every thread holds one frequency, so the rotation needs no shared cos/sin row; the new key
//    (rotated in fp64 from the handle's cos/sin table and rounded once to bf16, the bits
//    ham_kv_append stores) and the rotated query heads of the group go to shared memory;
//  - a warp per query head: lane pair j scores slot j, half of head_dim each, so that all scores
//    take one short dot product and one shuffle, the softmax (fp32, exact exp) four shuffles twice;
//    the weighted sum of values stays in registers.
// A call of the layers of a batch of 8 in turn (32/8 heads of 64): 6.0 us before (every load after
// the wait in two round trips, scores one after the other with five shuffles each), 3.5 us now.
#include <cuda_bf16.h>

#include "ham_micro.cuh"
#include "ham_ptx.cuh"

namespace ham {
namespace {

constexpr int kMicroThreads = 128;
constexpr int kMicroWarps = kMicroThreads / 32;

__device__ __forceinline__ float bf16_value(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }
__device__ __forceinline__ double bf16_value_d(uint16_t b) { return (double)bf16_value(b); }
__device__ __forceinline__ uint16_t to_bf16_bits(double x) {
  return __bfloat16_as_ushort(__double2bfloat16(x));
}

template <int D>
__global__ void __launch_bounds__(kMicroThreads) micro_step_kernel(MicroView v) {
  constexpr int HALF = D / 2;
  constexpr int PER = D / 32;        // output elements per lane
  constexpr int VEC = D / 8;         // 16-byte pieces of a row
  constexpr int ROW = D + 8;         // row stride of the key and value tiles (bank spread)
  constexpr int kPairs = (9 * HALF + kMicroThreads - 1) / kMicroThreads;  // pairs a thread, at most
  static_assert(kMicroThreads % HALF == 0, "a thread's pairs share one frequency");
  const int b = blockIdx.x, g = blockIdx.y, tid = threadIdx.x;
  const int G = v.n_q_heads / v.n_kv_heads;
  const int Hkv = v.n_kv_heads;
  const int warp = tid >> 5, lane = tid & 31;
  const int freq = tid % HALF;
  __shared__ __align__(16) uint16_t ks[kMicroMaxSlots][ROW];
  __shared__ __align__(16) uint16_t vs[kMicroMaxSlots][ROW];
  __shared__ __align__(16) float qs[8][D];        // the group's query heads (bf16 values)

  if (!v.early) grid_dependency_wait();
  // Library state: the counters and the page entry, then the old entries and the cos/sin at the
  // position unless the caller gives it.
  const int32_t n = v.num_slots[b];
  int64_t page = v.page_table[(int64_t)b * v.max_pages];   // the sequence's only page
  int64_t p = v.pos_mode == HAM_POS_SLOT ? (int64_t)n : v.num_tokens[b];
  const int64_t tokens = g == 0 && tid == 0 ? v.num_tokens[b] : 0;
  const bool page_ok = page >= 0 && page < v.pool_pages;
  const bool n_ok = n >= 0 && n < v.max_slots;
  if (!page_ok) page = 0;
  // (a bad page: nothing readable, the sequence attends over no slot)
  const int old = !page_ok || n < 0 ? 0 : (n > v.max_slots ? v.max_slots : n);
  const int64_t row0 = (page * Hkv + g) * v.page_slots;    // row of slot 0, this KV head
  for (int idx = tid; idx < old * VEC; idx += kMicroThreads) {
    const int j = idx / VEC, e = idx % VEC;
    const uint4 kx = reinterpret_cast<const uint4 *>(v.k_pool + (row0 + j) * D)[e];
    const uint4 vx = reinterpret_cast<const uint4 *>(v.v_pool + (row0 + j) * D)[e];
    *reinterpret_cast<uint4 *>(&ks[j][8 * e]) = kx;
    *reinterpret_cast<uint4 *>(&vs[j][8 * e]) = vx;
  }
  double2 cs = make_double2(1.0, 0.0);
  auto turn_at = [&](int64_t at) {
    if (at >= 0 && at < v.rope_positions) return v.rope_table[at * HALF + freq];
    double c, sn;
    sincos((double)at * v.inv_freq[freq], &sn, &c);
    return make_double2(c, sn);
  };
  if (!v.pos && n_ok) cs = turn_at(p);
  if (v.early) grid_dependency_wait();
  grid_launch_dependents();

  // The caller's inputs: this thread's pairs of the query heads (rows 0 .. G-1) and the new key
  // (row G), a piece of the new value, the token count and perhaps the position.
  const uint16_t *q_src = v.q + ((int64_t)b * v.n_q_heads + (int64_t)g * G) * D;
  const int64_t kv_off = ((int64_t)b * Hkv + g) * D;
  uint16_t lo[kPairs], hi[kPairs];
#pragma unroll
  for (int x = 0; x < kPairs; ++x) {
    const int r = (tid + x * kMicroThreads) / HALF;
    lo[x] = hi[x] = 0;
    if (r <= G) {
      const uint16_t *src = r < G ? q_src + r * D : v.k_new + kv_off;
      lo[x] = src[freq];
      hi[x] = src[freq + HALF];
    }
  }
  uint4 vn = make_uint4(0, 0, 0, 0);
  if (tid < VEC) vn = reinterpret_cast<const uint4 *>(v.v_new + kv_off)[tid];
  const int32_t t = v.ntok[b];
  int32_t err = 0;
  if (t < 1) err = HAM_DEVERR_NTOK;
  else if (!n_ok) err = n < 0 ? HAM_DEVERR_SLOTS : HAM_DEVERR_CAPACITY;
  else if (!page_ok) err = HAM_DEVERR_PAGE;
  const bool ok = err == 0;
  if (err && g == 0 && tid == 0) record_error(v.err, err);
  if (v.pos) {
    p = v.pos[b];
    if (ok) cs = turn_at(p);
  }
  // the cluster's CTAs have read the counter once they have all arrived
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");

  // Turn the pairs: x0 c - x1 s, x1 c + x0 s in fp64 with explicit _rn operations (no contraction),
  // rounded once to bf16.
#pragma unroll
  for (int x = 0; x < kPairs; ++x) {
    const int r = (tid + x * kMicroThreads) / HALF;
    if (r > G) continue;
    uint16_t y0 = lo[x], y1 = hi[x];
    if (ok) {
      const double x0 = bf16_value_d(lo[x]), x1 = bf16_value_d(hi[x]);
      y0 = to_bf16_bits(__dsub_rn(__dmul_rn(x0, cs.x), __dmul_rn(x1, cs.y)));
      y1 = to_bf16_bits(__dadd_rn(__dmul_rn(x1, cs.x), __dmul_rn(x0, cs.y)));
    }
    if (r < G) {
      qs[r][freq] = bf16_value(y0);
      qs[r][freq + HALF] = bf16_value(y1);
      if (ok && v.q_rot) {
        uint16_t *dst = v.q_rot + ((int64_t)b * v.n_q_heads + (int64_t)g * G + r) * D;
        dst[freq] = y0;
        dst[freq + HALF] = y1;
      }
    } else if (ok) {  // the new key's row
      uint16_t *dst = v.k_pool + (row0 + n) * D;
      ks[n][freq] = dst[freq] = y0;
      ks[n][freq + HALF] = dst[freq + HALF] = y1;
    }
  }
  if (ok && tid < VEC) {
    *reinterpret_cast<uint4 *>(&vs[n][8 * tid]) = vn;
    reinterpret_cast<uint4 *>(v.v_pool + (row0 + n) * D)[tid] = vn;
  }
  __syncthreads();

  // attention of the group's query heads over the L entries, one warp per head; lanes 2 j, 2 j + 1
  // score slot j
  const int L = ok ? n + 1 : old;
  const float scale = rsqrtf((float)D);
  const int slot = lane >> 1, part = (lane & 1) * HALF;
  for (int hl = warp; hl < G; hl += kMicroWarps) {
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int e = 0; e < HALF; e += 8) {
      const uint4 kx = *reinterpret_cast<const uint4 *>(&ks[slot][part + e]);
      const float4 qa = *reinterpret_cast<const float4 *>(&qs[hl][part + e]);
      const float4 qb = *reinterpret_cast<const float4 *>(&qs[hl][part + e + 4]);
      s0 = fmaf(qa.x, __uint_as_float(kx.x << 16), s0);
      s1 = fmaf(qa.y, __uint_as_float(kx.x & 0xFFFF0000u), s1);
      s0 = fmaf(qa.z, __uint_as_float(kx.y << 16), s0);
      s1 = fmaf(qa.w, __uint_as_float(kx.y & 0xFFFF0000u), s1);
      s0 = fmaf(qb.x, __uint_as_float(kx.z << 16), s0);
      s1 = fmaf(qb.y, __uint_as_float(kx.z & 0xFFFF0000u), s1);
      s0 = fmaf(qb.z, __uint_as_float(kx.w << 16), s0);
      s1 = fmaf(qb.w, __uint_as_float(kx.w & 0xFFFF0000u), s1);
    }
    float sc = s0 + s1;
    sc += __shfl_xor_sync(kFull, sc, 1);
    sc = slot < L ? sc * scale : -INFINITY;  // (rows past L hold whatever shared memory did)
    float m = sc;
#pragma unroll
    for (int o = 2; o < 32; o <<= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    const float w = slot < L ? expf(sc - m) : 0.f;
    float l = w;
#pragma unroll
    for (int o = 2; o < 32; o <<= 1) l += __shfl_xor_sync(kFull, l, o);
    float acc[PER];
#pragma unroll
    for (int e = 0; e < PER; ++e) acc[e] = 0.f;
#pragma unroll 4
    for (int j = 0; j < L; ++j) {
      const float wj = __shfl_sync(kFull, w, 2 * j);
#pragma unroll
      for (int e = 0; e < PER; ++e) acc[e] = fmaf(wj, bf16_value(vs[j][lane * PER + e]), acc[e]);
    }
    const float inv = L > 0 ? 1.f / l : 0.f;
    const int64_t o = ((int64_t)b * v.n_q_heads + (int64_t)g * G + hl) * D + lane * PER;
    if (v.out_f32) {
      float *dst = static_cast<float *>(v.out) + o;
#pragma unroll
      for (int e = 0; e < PER; ++e) dst[e] = acc[e] * inv;
    } else {
      uint16_t *dst = static_cast<uint16_t *>(v.out) + o;
#pragma unroll
      for (int e = 0; e < PER; ++e) dst[e] = __bfloat16_as_ushort(__float2bfloat16_rn(acc[e] * inv));
    }
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (ok && g == 0 && tid == 0) {  // rank 0 advances the counters
    const int64_t meta = page * v.page_slots + n;
    v.slot_pos[meta] = (int32_t)p;
    v.slot_ntok[meta] = t;
    v.num_slots[b] = n + 1;
    v.num_tokens[b] = tokens + t;
  }
}

template <int D>
cudaError_t launch_d(const MicroView &v, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)v.batch, (unsigned)v.n_kv_heads);
  cfg.blockDim = dim3(kMicroThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1;
  attr[1].val.clusterDim.y = (unsigned)v.n_kv_heads;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, micro_step_kernel<D>, v);
}

}  // namespace

cudaError_t launch_micro(const MicroView &v, cudaStream_t stream) {
  return v.head_dim == 64 ? launch_d<64>(v, stream) : launch_d<128>(v, stream);
}

}  // namespace ham
