// Order, statistics and prefix sums of ONE large instance with the whole GPU.
//
// The batch kernel (kvs_sort.cu) gives an instance to one CTA; for a sweep, which has a single instance, that
// left 147 SMs idle (4.5 ms for a million jobs, and 1.4 ms for the prefix sums on one CTA).  Here the jobs are cut
// into chunks of ORD_CHUNK, one CTA each: per radix pass (8-bit digits, least significant first) the chunks count
// their digits, one CTA per digit turns the counts into first positions (equal digits keep the order of the
// chunks), and the chunks place their jobs.  Index and key travel together as one 64-bit record, so that no
// pass looks a key up; the last pass writes the sorted lengths instead.  The work is small (a million jobs: about
// 60 MB moved, two passes); what bounds it is the length of the launches' chain, so the host reads the largest key
// back with the sizes and launches only the passes that are needed.
#include "kvs_internal.cuh"

namespace {

constexpr int OT = 1024;
constexpr int OWARPS = OT / 32;
constexpr int ORD_TILES = 4;
constexpr int ORD_CHUNK = OT * ORD_TILES;

// s_max, o_max and input checks of the jobs [job_off[0], job_off[1]) into info->stats (zeroed by the caller),
// and the range itself.
__global__ void __launch_bounds__(256) k_order_info(const i64* job_off, const int32_t* s, const int32_t* o, i64 n_total, i64 max_jobs, OrderInfo* info) {
  __shared__ int red[32];
  const i64 lo = job_off[0], hi = job_off[1];
  const bool fits = lo >= 0 && hi >= lo && hi <= n_total && hi - lo <= max_jobs;
  if (blockIdx.x == 0 && threadIdx.x == 0) { info->lo = lo; info->hi = hi; }
  if (!fits) return;
  int s_max = 0, o_max = 0, bad = 0;
  for (i64 j = lo + static_cast<i64>(blockIdx.x) * 256 + threadIdx.x; j < hi; j += static_cast<i64>(gridDim.x) * 256) {
    const int sv = s[j], ov = o[j];
    s_max = max(s_max, sv); o_max = max(o_max, ov);
    bad |= (sv < 0) | (ov < 1);
  }
  s_max = block_max(s_max, red, 0);
  o_max = block_max(o_max, red, 0);
  bad = block_max(bad, red, 0);
  if (threadIdx.x == 0) {
    atomicMax(&info->stats.s_max, s_max);
    atomicMax(&info->stats.o_max, o_max);
    if (bad) atomicOr(&info->stats.flags, static_cast<int>(KVS_EVAL_BAD_INPUT));
  }
}

__device__ __forceinline__ u32 digit_of(u32 key, int pass) { return (key >> (8 * pass)) & 255u; }

// counts[digit * n_chunks + chunk] of pass `pass`
__global__ void __launch_bounds__(OT) k_order_count(const int32_t* o, const u64* rec, i64 n, int pass, u32* counts) {
  __shared__ u32 hist[256];
  for (int i = threadIdx.x; i < 256; i += OT) hist[i] = 0;
  __syncthreads();
  const i64 j0 = static_cast<i64>(blockIdx.x) * ORD_CHUNK;
#pragma unroll
  for (int t = 0; t < ORD_TILES; ++t) {
    const i64 j = j0 + t * OT + threadIdx.x;
    if (j < n) {
      const u32 key = pass == 0 ? static_cast<u32>(o[j]) : static_cast<u32>(rec[j] >> 32);
      atomicAdd(&hist[digit_of(key, pass)], 1u);
    }
  }
  __syncthreads();
  for (int d = threadIdx.x; d < 256; d += OT) counts[static_cast<i64>(d) * gridDim.x + blockIdx.x] = hist[d];
}

// Per digit (one CTA each): exclusive scan of the chunks' counts in place, and the digit's total.
__global__ void __launch_bounds__(256) k_order_scan(u32* counts, i64 chunks, u32* total) {
  __shared__ u32 wsum[8];
  const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
  u32* const row = counts + static_cast<i64>(blockIdx.x) * chunks;
  u32 run = 0;
  for (i64 c0 = 0; c0 < chunks; c0 += 256) {
    const i64 c = c0 + tid;
    const u32 v = c < chunks ? row[c] : 0u;
    const u32 incl = warp_incl(v);
    __syncthreads();
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    const u32 w = lane < 8 ? wsum[lane] : 0u;
    const u32 wi = warp_incl(w);
    const u32 before = __shfl_sync(0xffffffffu, wi - w, warp);      // all lanes take part in the shuffle
    if (c < chunks) row[c] = run + before + incl - v;
    run += __shfl_sync(0xffffffffu, wi, 7);
  }
  if (tid == 0) total[blockIdx.x] = run;
}

// Places the jobs of a chunk.  Stable: lanes with equal digits rank by lane, warps and tiles in order behind the
// running position of the digit.
__global__ void __launch_bounds__(OT) k_order_place(const int32_t* s, const int32_t* o, const u64* src, u64* dst, i64 n, int pass, int last,
                                                    const u32* first, const u32* total, int32_t* sorted_s, int32_t* sorted_o) {
  extern __shared__ u32 dyn[];
  u32 (*const warp_cnt)[256] = reinterpret_cast<u32 (*)[256]>(dyn);
  const int tid = threadIdx.x, warp = tid >> 5;
  for (int i = tid; i < OWARPS * 256; i += OT) dyn[i] = 0;
  __shared__ u32 wsum[8];
  // first position of this chunk's jobs of digit `tid`: jobs of smaller digits, then those of earlier chunks
  u32 bucket = 0;
  if (tid < 256) {
    const u32 v = total[tid], incl = warp_incl(v);
    if (lane_id() == 31) wsum[warp] = incl;
    bucket = incl - v + first[static_cast<i64>(tid) * gridDim.x + blockIdx.x];
  }
  __syncthreads();
  if (tid < 256) for (int w = 0; w < warp; ++w) bucket += wsum[w];
  const i64 j0 = static_cast<i64>(blockIdx.x) * ORD_CHUNK;
  u64 rec[ORD_TILES];
#pragma unroll
  for (int t = 0; t < ORD_TILES; ++t) {
    const i64 j = j0 + t * OT + tid;
    rec[t] = 0;
    if (j < n) rec[t] = pass == 0 ? (static_cast<u64>(static_cast<u32>(o[j])) << 32 | static_cast<u32>(j)) : src[j];
  }
#pragma unroll
  for (int t = 0; t < ORD_TILES; ++t) {
    const bool valid = j0 + t * OT + tid < n;
    const u32 digit = valid ? digit_of(static_cast<u32>(rec[t] >> 32), pass) : 256u;
    const u32 peers = __match_any_sync(0xffffffffu, digit);
    const u32 rank = __popc(peers & lanemask_lt());
    const bool leader = valid && rank == 0;
    if (leader) warp_cnt[warp][digit] = __popc(peers);
    __syncthreads();
    if (tid < 256) {
#pragma unroll 8
      for (int w = 0; w < OWARPS; ++w) { const u32 c = warp_cnt[w][tid]; warp_cnt[w][tid] = bucket; bucket += c; }
    }
    __syncthreads();
    if (valid) {
      const u32 pos = warp_cnt[warp][digit] + rank;
      if (last) {
        sorted_o[pos] = static_cast<int32_t>(rec[t] >> 32);
        sorted_s[pos] = s[static_cast<u32>(rec[t])];
      } else {
        dst[pos] = rec[t];
      }
    }
    __syncthreads();
    for (int i = tid; i < OWARPS * 256; i += OT) dyn[i] = 0;     // the column scan turned every count into a position
    __syncthreads();
  }
}

// Sums of s and o per chunk; exclusive scan of those sums; prefix sums inside the chunks.
__global__ void __launch_bounds__(OT) k_prefix_sums(const int32_t* s, const int32_t* o, i64 n, i64* part) {
  __shared__ i64 red[32];
  const i64 j0 = static_cast<i64>(blockIdx.x) * ORD_CHUNK;
  i64 vs = 0, vo = 0;
#pragma unroll
  for (int t = 0; t < ORD_TILES; ++t) {
    const i64 j = j0 + t * OT + threadIdx.x;
    if (j < n) { vs += s[j]; vo += o[j]; }
  }
  vs = block_sum(vs, red);
  vo = block_sum(vo, red);
  if (threadIdx.x == 0) { part[2 * static_cast<i64>(blockIdx.x)] = vs; part[2 * static_cast<i64>(blockIdx.x) + 1] = vo; }
}

__global__ void __launch_bounds__(64) k_prefix_scan(i64* part, i64 chunks) {
  // warp 0 scans the sums of s, warp 1 those of o
  const int which = threadIdx.x >> 5, lane = lane_id();
  i64 run = 0;
  for (i64 c0 = 0; c0 < chunks; c0 += 32) {
    const i64 c = c0 + lane;
    const i64 v = c < chunks ? part[2 * c + which] : 0;
    const i64 incl = warp_incl(v);
    if (c < chunks) part[2 * c + which] = run + incl - v;
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
}

__global__ void __launch_bounds__(OT) k_prefix_apply(const int32_t* s, const int32_t* o, i64 n, const i64* part, i64* ps, u32* ps32, i64* po) {
  __shared__ i64 ws[32], wo[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
  // `part` NULL: a single chunk
  i64 run_s = part ? part[2 * static_cast<i64>(blockIdx.x)] : 0, run_o = part ? part[2 * static_cast<i64>(blockIdx.x) + 1] : 0;
  if (blockIdx.x == 0 && tid == 0) { ps[0] = 0; ps32[0] = 0; po[0] = 0; }
  const i64 j0 = static_cast<i64>(blockIdx.x) * ORD_CHUNK + static_cast<i64>(tid) * ORD_TILES;
  i64 vs[ORD_TILES], vo[ORD_TILES], ts = 0, to = 0;
#pragma unroll
  for (int t = 0; t < ORD_TILES; ++t) {
    ts += j0 + t < n ? s[j0 + t] : 0; to += j0 + t < n ? o[j0 + t] : 0;
    vs[t] = ts; vo[t] = to;
  }
  const i64 is = warp_incl(ts), io = warp_incl(to);
  if (lane == 31) { ws[warp] = is; wo[warp] = io; }
  __syncthreads();
  const i64 a = ws[lane], b = wo[lane];
  const i64 ia = warp_incl(a), ib = warp_incl(b);
  run_s += __shfl_sync(0xffffffffu, ia - a, warp) + is - ts;
  run_o += __shfl_sync(0xffffffffu, ib - b, warp) + io - to;
#pragma unroll
  for (int t = 0; t < ORD_TILES; ++t)
    if (j0 + t < n) { ps[j0 + t + 1] = run_s + vs[t]; ps32[j0 + t + 1] = static_cast<u32>(run_s + vs[t]); po[j0 + t + 1] = run_o + vo[t]; }
}

}  // namespace

i64 kvs_order_chunks(i64 n) { return (n + ORD_CHUNK - 1) / ORD_CHUNK; }

cudaError_t kvs_launch_order_info(const i64* job_off, const int32_t* s, const int32_t* o, i64 n_total, i64 max_jobs, OrderInfo* info, int sm_count, cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(info, 0, sizeof(OrderInfo), stream);
  if (e != cudaSuccess) return e;
  const i64 want = (max_jobs + 2047) / 2048, most = static_cast<i64>(sm_count) * 4;
  k_order_info<<<static_cast<unsigned>(want < 1 ? 1 : (want < most ? want : most)), 256, 0, stream>>>(job_off, s, o, n_total, max_jobs, info);
  return cudaGetLastError();
}

// s, o: the instance's own jobs.  rec0, rec1: n records each; counts: 256 * (kvs_order_chunks(n) + 1) words.
cudaError_t kvs_launch_order(const int32_t* s, const int32_t* o, i64 n, int o_max, u64* rec0, u64* rec1, u32* counts,
                             int32_t* sorted_s, int32_t* sorted_o, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  constexpr int smem = OWARPS * 256 * 4;
  const unsigned chunks = static_cast<unsigned>(kvs_order_chunks(n));
  int passes = 1;
  while (passes < 4 && (static_cast<u32>(o_max) >> (8 * passes)) != 0) ++passes;
  u64* buf[2] = {rec0, rec1};
  u32* const total = counts + static_cast<i64>(256) * chunks;
  for (int pass = 0; pass < passes; ++pass) {
    const u64* const src = buf[(pass + 1) & 1];
    k_order_count<<<chunks, OT, 0, stream>>>(o, src, n, pass, counts);
    k_order_scan<<<256, 256, 0, stream>>>(counts, chunks, total);
    k_order_place<<<chunks, OT, smem, stream>>>(s, o, src, buf[pass & 1], n, pass, pass == passes - 1, counts, total, sorted_s, sorted_o);
  }
  return cudaGetLastError();
}

// Exclusive prefix sums of s and o in key order (n + 1 entries each); part: 2 * kvs_order_chunks(n) entries.
cudaError_t kvs_launch_prefix(const int32_t* sorted_s, const int32_t* sorted_o, i64 n, i64* part, i64* prefix_s, u32* prefix_s32, i64* prefix_o, cudaStream_t stream) {
  const unsigned chunks = static_cast<unsigned>(n > 0 ? kvs_order_chunks(n) : 1);
  if (chunks > 1) {
    k_prefix_sums<<<chunks, OT, 0, stream>>>(sorted_s, sorted_o, n, part);
    k_prefix_scan<<<1, 64, 0, stream>>>(part, chunks);
  }
  k_prefix_apply<<<chunks, OT, 0, stream>>>(sorted_s, sorted_o, n, chunks > 1 ? part : nullptr, prefix_s, prefix_s32, prefix_o);
  return cudaGetLastError();
}
