// Per-instance statistics and the stable order of jobs by (estimated) response length.
//
// One CTA handles one instance at a time.  It first reduces the instance's statistics
// (largest prompt, response and key; input validation), then, window by window, sorts the
// job indices by key with a least-significant-digit radix sort (8-bit digits).  Stability
// (ties keep the original index order) is what makes the order unique, so that the per-job
// results agree bit for bit with a stable comparison sort.
//
// Each pass ranks one tile of TILE_N jobs at a time.  A warp takes 32 * ITEMS consecutive ones, row by row: lanes with equal
// digits find each other with a warp match and stand behind what the warp has counted so far of their digit in its row of counters
// in shared memory; one column scan per tile, eight counters a thread, turns the counters into offsets behind the running
// bucket position.  Two block barriers per tile.  Only 4 bytes per job move per pass: the index, together with the key in the
// upper half of the word when both fit 16 bits; otherwise the next pass re-reads the key through the index.
//
// What bounds it: latencies - of the loads (DRAM and L2), of the match chains and at the barriers - and the scattered 4-byte stores, not
// bandwidth (32 bytes a job must move, some 60 do).  More instances in flight do not help, their arrays leave the L2: 2,048 instances of
// 50,000 jobs take 3.04 ms with two CTAs of 512 threads and four jobs a thread and tile per SM, 3.75 with four of them, 3.9 with three and
// eight jobs a thread, 3.4 with one of 1,024 threads (two of 1,024 threads and one job a thread and tile: 3.42).
#include "kvs_internal.cuh"

namespace {

constexpr int T = KVS_SORT_THREADS;
constexpr int WARPS = T / 32;
constexpr int ITEMS = KVS_SORT_ITEMS;
constexpr int TILE_N = T * ITEMS;
constexpr int PER_DIGIT = T / 256;                       // threads that scan the column of one digit
constexpr int ROWS = WARPS / PER_DIGIT;                  // counters each of them takes
// Words per row of counters: the PER_DIGIT threads of a digit and those of its neighbours fall into different banks.
constexpr int ROW_W = 256 + (PER_DIGIT == 4 ? 1 : 2);
static_assert(PER_DIGIT >= 1 && PER_DIGIT <= 4 && ROWS == 8, "column scan");

__device__ __forceinline__ int32_t key_at(const SortParams& p, i64 lo, int idx) {
  return p.key ? p.key[lo + idx] : p.o[lo + idx];
}

// Counts the digits of a key; most keys have 0 as their second digit and above (of a warp's keys one addition books them).
__device__ __forceinline__ void count_digits(u32 (*hist)[256], u32 key, bool valid, int first, int passes) {
  for (int d = first; d < passes; ++d) {
    const u32 digit = (key >> (8 * d)) & 255u;
    if (d == 0) {
      if (valid) atomicAdd(&hist[0][digit], 1u);
    } else {
      const u32 zeros = __ballot_sync(0xffffffffu, valid && digit == 0);
      if (lane_id() == 0 && zeros) atomicAdd(&hist[d][0], static_cast<u32>(__popc(zeros)));
      if (valid && digit != 0) atomicAdd(&hist[d][digit], 1u);
    }
  }
}

// Sort positions [seg_lo, seg_hi) of the instance starting at global job index lo.  The last pass
// holds every job's key when it places the job, so it also writes the keys in sorted order (one more
// scattered store that merges in L2 like the index, instead of a gather afterwards); returns
// whether it did.
// packed: indices and keys are below 2^16, so a pass that is not the last stores (key << 16 | index)
// and the next pass needs no look-up of the key through the index.
// counted: hist holds the counts of the first that many digits.
__device__ __forceinline__ bool sort_segment(const SortParams& p, i64 lo, int seg_lo, int seg_hi, int passes, bool packed, int counted,
                             u32* counters, u32 (*hist)[256]) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
  const int n = seg_hi - seg_lo;
  int32_t* const out = p.perm + lo + seg_lo;
  if (passes == 0 || n <= 1) {
    for (int j = tid; j < n; j += T) out[j] = seg_lo + j;
    __syncthreads();
    return false;
  }
  // digit histograms of the passes that are not counted yet, in one sweep
  u32* const row = counters + warp * ROW_W;
  for (int d = lane; d < 256; d += 32) row[d] = 0;         // stays zero between tiles, see below
  if (counted < passes) {
    for (int i = tid + counted * 256; i < passes * 256; i += T) (&hist[0][0])[i] = 0;
    __syncthreads();
    for (int j0 = 0; j0 < n; j0 += T) {
      const int j = j0 + tid;
      count_digits(hist, j < n ? static_cast<u32>(key_at(p, lo, seg_lo + j)) : 0u, j < n, counted, passes);
    }
  }
  __syncthreads();
  // exclusive scan of each histogram: warp d scans histogram d, 8 digits per lane
  if (warp < passes) {
    u32 v[8], sum = 0;
    for (int i = 0; i < 8; ++i) { v[i] = hist[warp][lane * 8 + i]; sum += v[i]; }
    u32 run = warp_incl(sum) - sum;
    for (int i = 0; i < 8; ++i) { hist[warp][lane * 8 + i] = run; run += v[i]; }
  }
  __syncthreads();

  for (int pass = 0; pass < passes; ++pass) {
    // the last pass must land in perm: passes alternate between the two buffers
    const bool to_perm = ((passes - 1 - pass) & 1) == 0;
    int32_t* dst = (to_perm ? p.perm : p.perm_tmp) + lo + seg_lo;
    const int32_t* src = (to_perm ? p.perm_tmp : p.perm) + lo + seg_lo;
    int32_t* const key_dst = pass == passes - 1 ? (p.key ? p.sorted_key : p.sorted_o) + lo + seg_lo : nullptr;
    const int shift = 8 * pass;
    for (int j0 = 0; j0 < n; j0 += TILE_N) {
      const int jw = j0 + warp * (32 * ITEMS) + lane;
      int idx[ITEMS];
      u32 key[ITEMS], rank[ITEMS];
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const int j = jw + 32 * i;
        idx[i] = seg_lo + j;
        key[i] = 0;
        if (j < n) {
          if (pass == 0) key[i] = static_cast<u32>(key_at(p, lo, idx[i]));
          else idx[i] = src[j];
        }
      }
      if (pass > 0) {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
          if (packed) { key[i] = static_cast<u32>(idx[i]) >> 16; idx[i] &= 0xffff; }
          else if (jw + 32 * i < n) key[i] = static_cast<u32>(key_at(p, lo, idx[i]));
        }
      }
      // rank among the warp's jobs of the same digit, in order
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const bool valid = jw + 32 * i < n;
        const u32 digit = valid ? (key[i] >> shift) & 255u : 256u;     // jobs past the end keep to themselves
        const u32 peers = __match_any_sync(0xffffffffu, digit);
        const u32 below = __popc(peers & lanemask_lt());
        const u32 before = valid ? row[digit] : 0u;
        rank[i] = before + below;
        __syncwarp();
        if (valid && below == 0) row[digit] = before + __popc(peers);
        __syncwarp();
      }
      __syncthreads();
      {
        const int digit = tid / PER_DIGIT, part = tid % PER_DIGIT;
        u32* const column = counters + part * ROWS * ROW_W + digit;
        u32 c[ROWS], sum = 0;
#pragma unroll
        for (int i = 0; i < ROWS; ++i) { c[i] = column[i * ROW_W]; sum += c[i]; }
        u32 incl = sum;
#pragma unroll
        for (int d = 1; d < PER_DIGIT; d <<= 1) {
          const u32 y = __shfl_up_sync(0xffffffffu, incl, d);
          if (part >= d) incl += y;
        }
        u32 at = hist[pass][digit] + incl - sum;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < ROWS; ++i) { column[i * ROW_W] = at; at += c[i]; }
        if (part == PER_DIGIT - 1) hist[pass][digit] = at;               // running position of the digit
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        if (jw + 32 * i < n) {
          const u32 pos = row[(key[i] >> shift) & 255u] + rank[i];
          dst[pos] = (packed && !key_dst) ? static_cast<int32_t>(key[i] << 16 | static_cast<u32>(idx[i])) : idx[i];
          if (key_dst) key_dst[pos] = static_cast<int32_t>(key[i]);
        }
      }
      // the row is the warp's own again until the next tile's barrier
      __syncwarp();
#pragma unroll
      for (int d = 0; d < 8; ++d) row[32 * d + lane] = 0;
      __syncwarp();
    }
    __syncthreads();   // the next pass reads what this one stored
  }
  return true;
}

__global__ void __launch_bounds__(KVS_SORT_THREADS, KVS_SORT_CTAS) k_stats_sort(SortParams p) {
  extern __shared__ __align__(16) u32 counters[];
  __shared__ u32 hist[4][256];
  __shared__ int red[32];
  __shared__ i64 wsum[32];
  __shared__ int seg_end;
  const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();

  // Windows are ordered independently: a batch of few instances with windows gives each of them to several CTAs (parts), which
  // take its windows in turn; each forms the statistics it needs by itself.
  const int parts = p.parts;
  for (i64 item = blockIdx.x; item < p.n_instances * parts; item += gridDim.x) {
    const i64 inst = item / parts;
    const int part = static_cast<int>(item % parts);
    const i64 lo = p.job_off[inst], hi = p.job_off[inst + 1];
    int flags = 0;
    if (hi < lo || hi - lo > p.max_jobs) flags = KVS_EVAL_BAD_INPUT;
    const int n = flags ? 0 : static_cast<int>(hi - lo);
    // an instance that is ordered as a whole has the first two digits of its keys counted on the way
    const bool windows = p.window > 0 && p.arrival;
    const bool count = p.need_order && !windows;
    if (count) {
      __syncthreads();
      for (int i = tid; i < 512; i += T) (&hist[0][0])[i] = 0;
      __syncthreads();
    }
    int s_max = 0, o_max = 0, key_max = 0, bad = 0;
    constexpr int U = 4;
    for (int j0 = 0; j0 < n; j0 += U * T) {
      int sv[U], ov[U], kv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j0 + u * T + tid;
        sv[u] = j < n ? p.s[lo + j] : 0;
        ov[u] = j < n ? p.o[lo + j] : 1;
        kv[u] = p.key && j < n ? p.key[lo + j] : ov[u];
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j0 + u * T + tid;
        if (j < n) { s_max = max(s_max, sv[u]); o_max = max(o_max, ov[u]); key_max = max(key_max, kv[u]); }
        bad |= (sv[u] < 0) | (ov[u] < 1) | (kv[u] < 1);
        if (count) count_digits(hist, static_cast<u32>(kv[u]), j < n, 0, 2);
        if (p.arrival && j < n) {
          const i64 a = p.arrival[lo + j];
          bad |= (a < 0) | (j > 0 && p.arrival[lo + j - 1] > a);
        }
      }
    }
    s_max = block_max(s_max, red, 0);
    o_max = block_max(o_max, red, 0);
    key_max = block_max(key_max, red, 0);
    bad = block_max(bad, red, 0);
    if (bad) flags = KVS_EVAL_BAD_INPUT;
    if (tid == 0 && part == 0) p.stats[inst] = InstStats{s_max, o_max, key_max, flags};
    if (!p.need_order || flags) continue;  // uniform across the CTA

    const int passes = key_max > 0 ? (32 - __clz(key_max) + 7) / 8 : 0;
    int seg_lo = 0;
    for (int w = 0; seg_lo < n; ++w) {
      if (tid < 32) {
        const int end = windows ? window_end(p.arrival + lo, seg_lo, n, p.window) : n;
        if (tid == 0) seg_end = end;
      }
      __syncthreads();
      const int seg_hi = seg_end;
      if (w % parts != part) {
        __syncthreads();
        seg_lo = seg_hi;
        continue;
      }
      const bool have_key = sort_segment(p, lo, seg_lo, seg_hi, passes, n <= 65536 && key_max < 65536, count ? min(passes, 2) : 0, counters, hist);
      __syncthreads();
      for (int j0 = seg_lo + tid; j0 < seg_hi; j0 += U * T) {
        int idx[U], sv[U], ov[U], kv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) idx[u] = j0 + u * T < seg_hi ? p.perm[lo + j0 + u * T] : seg_lo;
        // streaming stores: read back much later, by another kernel
#pragma unroll
        for (int u = 0; u < U; ++u) {
          sv[u] = p.s[lo + idx[u]];
          ov[u] = p.key || !have_key ? p.o[lo + idx[u]] : 0;
          kv[u] = p.key && !have_key ? p.key[lo + idx[u]] : 0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int j = j0 + u * T;
          if (j < seg_hi) {
            __stcs(&p.sorted_s[lo + j], sv[u]);
            if (p.key || !have_key) __stcs(&p.sorted_o[lo + j], ov[u]);
            if (p.key && !have_key) __stcs(&p.sorted_key[lo + j], kv[u]);
            if (p.iperm) p.iperm[lo + idx[u]] = j;
          }
        }
      }
      __syncthreads();
      seg_lo = seg_hi;
    }
    if (p.prefix_s) {
      // exclusive prefix sums of s in schedule order (n + 1 entries per instance): the event form
      // of the peak reads the prompt tokens of any contiguous rank range as one difference
      i64* const ps = p.prefix_s + lo + inst;
      i64 run = 0;
      if (tid == 0) ps[0] = 0;
      for (int j0 = 0; j0 < n; j0 += TILE_N) {
        // a warp takes 32 * ITEMS consecutive ones, row by row
        const int jw = j0 + warp * (32 * ITEMS) + lane;
        u32 v[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) v[i] = jw + 32 * i < n ? static_cast<u32>(p.sorted_s[lo + jw + 32 * i]) : 0u;
        i64 total = 0;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) total += v[i];
        total = warp_sum(total);
        __syncthreads();
        if (lane == 0) wsum[warp] = total;
        __syncthreads();
        const i64 w = lane < WARPS ? wsum[lane] : 0;
        const i64 wi = warp_incl(w);
        i64 before = run + __shfl_sync(0xffffffffu, wi - w, warp);     // all lanes take part in the shuffle
        run += __shfl_sync(0xffffffffu, wi, 31);
        if (s_max < (1 << 26)) {                        // a row adds up in 32 bits
#pragma unroll
          for (int i = 0; i < ITEMS; ++i) {
            const u32 incl = warp_incl(v[i]);
            if (jw + 32 * i < n) __stcs(&ps[jw + 32 * i + 1], before + incl);
            before += __shfl_sync(0xffffffffu, incl, 31);
          }
        } else {
#pragma unroll
          for (int i = 0; i < ITEMS; ++i) {
            const i64 incl = warp_incl(static_cast<i64>(v[i]));
            if (jw + 32 * i < n) __stcs(&ps[jw + 32 * i + 1], before + incl);
            before += __shfl_sync(0xffffffffu, incl, 31);
          }
        }
      }
    }
  }
}

}  // namespace

namespace {

// Statistics alone (the same as the first part of k_stats_sort, which has a CTA per SM's worth of shared memory for
// the ordering and so few loads in flight): one CTA of 256 threads per instance, four jobs per thread in flight.
__global__ void __launch_bounds__(256) k_stats(SortParams p) {
  __shared__ int red[32];
  constexpr int U = 4;
  for (i64 inst = blockIdx.x; inst < p.n_instances; inst += gridDim.x) {
    const i64 lo = p.job_off[inst], hi = p.job_off[inst + 1];
    int flags = 0;
    if (hi < lo || hi - lo > p.max_jobs) flags = KVS_EVAL_BAD_INPUT;
    const int n = flags ? 0 : static_cast<int>(hi - lo);
    int s_max = 0, o_max = 0, bad = 0;
    for (int j0 = threadIdx.x; j0 < n; j0 += U * 256) {
      int sv[U], ov[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j0 + u * 256;
        sv[u] = j < n ? __ldg(p.s + lo + j) : 0;
        ov[u] = j < n ? __ldg(p.o + lo + j) : 1;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        s_max = max(s_max, sv[u]); o_max = max(o_max, ov[u]);
        bad |= (sv[u] < 0) | (ov[u] < 1);
      }
    }
    if (n == 0) o_max = 0;
    s_max = block_max(s_max, red, 0);
    o_max = block_max(o_max, red, 0);
    bad = block_max(bad, red, 0);
    if (bad) flags = KVS_EVAL_BAD_INPUT;
    if (threadIdx.x == 0) p.stats[inst] = InstStats{s_max, o_max, o_max, flags};
  }
}

}  // namespace

static constexpr size_t SORT_SMEM = WARPS * ROW_W * sizeof(u32);   // digit counts per warp

// Once per device, before the first launch.
cudaError_t kvs_setup_sort() {
  return cudaFuncSetAttribute(k_stats_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(SORT_SMEM));
}

// capacity: CTAs that the GPU holds at a time
cudaError_t kvs_launch_sort(const SortParams& p, int capacity, cudaStream_t stream) {
  if (p.n_instances <= 0) return cudaSuccess;
  if (!p.need_order && !p.key && !p.arrival) {
    const i64 most = static_cast<i64>(capacity) * 8;
    k_stats<<<static_cast<unsigned>(p.n_instances < most ? p.n_instances : most), 256, 0, stream>>>(p);
  } else {
    SortParams q = p;
    q.parts = 1;
    if (p.arrival && p.window > 0 && !p.prefix_s && p.n_instances < capacity) {
      const i64 g = capacity / p.n_instances;
      q.parts = static_cast<int>(g > 8 ? 8 : g);
    }
    const i64 items = p.n_instances * q.parts;
    k_stats_sort<<<static_cast<unsigned>(items < capacity ? items : capacity), KVS_SORT_THREADS, SORT_SMEM, stream>>>(q);
  }
  return cudaGetLastError();
}
