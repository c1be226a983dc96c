// Generic evaluator for explicit runs (the builder's run list or any user schedule).
//
// A run (start, len, s) holds s + u + 1 tokens in round start + u (Eq. Memory-Feasibility),
// i.e. c + t tokens in round t with c = s + 1 - start: it adds (c, 1) at `start` and (-c, -1) at `start + len` to two
// difference arrays, whose prefix sums A, B give memory(t) = A(t) + t * B(t).  Nothing is assumed about the order or
// overlap of the runs.
//
// k_tile_eval: one CTA per (evaluation, tile of rounds).  The CTA reads all runs of its evaluation (they stay in L2
// over the tiles), scatters the events of its rounds into difference arrays in shared memory and sums up, in registers, what
// the runs that cross its first round hold there, so the tiles do not depend on each other.  The sums over all runs are formed by the
// first tile alone, which leaves its flags to the last one.  It is bound by the visits of the runs (every tile looks at all of
// them) and shared-memory atomics; the 24 bytes per run and 4 per round that it has to move are a third of its time.  256
// schedules of 10,000 to 20,000 runs: a call of 123 us, 129 with every tile forming the sums; tiles of 27,648 rounds, one CTA of
// 1,024 threads per SM, which look at the runs half as often: 153.  With the arrays in global memory (k_generic_eval, four global
// atomics per run and 12 bytes of scratch per round to clear and re-read) the kernels alone took 142 us and 45 us.
// Arithmetic is modulo 2^32, exact as long as the sum of s + len over the runs, which bounds the memory of any round, is
// below 2^32; other evaluations (and ones with a negative s) are listed for k_generic_eval, which works in 64 bits.
#include <atomic>
#include <cstdio>

#include "kvs_internal.cuh"

namespace {

constexpr int T = 512;
constexpr int ITEMS = 4;

// ---- one tile of rounds per CTA ---------------------------------------------------------------------

constexpr int TT = 512;
constexpr int TK = 23;                       // rounds per thread at most; odd, so that the threads' stretches hit different banks
constexpr int TILE_MAX = TT * TK;

// Clears the per-evaluation words of the tiled kernel and checks the offsets that map tiles to evaluations: where they are
// not monotone within the stated capacity, *odd is set and the 64-bit kernel, which looks at every evaluation's offsets
// by itself, takes the whole call.
__global__ void __launch_bounds__(256) k_tile_init(GenericParams p, i64 capacity_total) {
  const i64 e = static_cast<i64>(blockIdx.x) * 256 + threadIdx.x;
  if (e >= p.runs.P) return;
  p.tile_peak[e] = 0;
  p.tile_done[e] = 0;
  const i64 a = p.ev.profile_off[e], b = p.ev.profile_off[e + 1];
  if (a < 0 || b < a || b > capacity_total || (e == 0 && a != 0)) *p.odd = 1u;
}

// The last evaluation whose first tile is not after `item`: tiles of e are items poff[e] / tile + e and up.
__device__ __forceinline__ i64 eval_of_item(const i64* __restrict__ poff, i64 P, i64 tile, i64 item) {
  i64 a = 0, b = P;                          // first(a) <= item; first(b) > item or b = P
  while (b - a > 1) {
    const i64 step = (b - a + 31) / 32;
    const i64 e = a + (static_cast<i64>(lane_id()) + 1) * step;
    const bool in = e < b && __ldg(poff + e) / tile + e <= item;
    const int m = __popc(__ballot_sync(0xffffffffu, in));
    const i64 nb = a + (static_cast<i64>(m) + 1) * step;
    a += static_cast<i64>(m) * step;
    if (nb < b) b = nb;
  }
  return a;
}

__global__ void __launch_bounds__(TT, 2) k_tile_eval(GenericParams p) {
  extern __shared__ u32 dyn[];
  __shared__ i64 red64[32];
  __shared__ u64 redu[32];
  __shared__ u32 scanA[32], scanB[32];
  __shared__ int red32[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
  const kvs_runs& R = p.runs;
  if (*p.odd) return;
  const i64 tile = p.tile;
  const int per = static_cast<int>(tile / TT);          // rounds per thread, odd
  u32* const dA = dyn;
  u32* const dB = dyn + tile;
  const i64 e = eval_of_item(p.ev.profile_off, R.P, tile, blockIdx.x);
  const i64 pbase = p.ev.profile_off[e], cap = p.ev.profile_off[e + 1] - pbase;
  const i64 my = blockIdx.x - (pbase / tile + e), n_tiles = cap > tile ? (cap + tile - 1) / tile : 1;
  if (my < 0 || my >= n_tiles) return;
  const i64 t0 = my * tile, t1 = t0 + tile;
  for (int i = tid; i < 2 * static_cast<int>(tile); i += TT) dyn[i] = 0;
  const i64 r0 = R.run_off[e], r1 = R.run_off[e + 1];
  i64 steps = 0, hmax = 0, flow = 0;
  u64 total = 0;
  u32 A0 = 0, B0 = 0;                                    // held in round t0 by runs that started before it
  int flags = 0;                                         // 1: bad input, 2: beyond the capacity, 4: not for 32 bits
  int last = 0;                                          // rounds of the tile up to the last run end
  const bool first = my == 0;                            // this tile forms what concerns all runs alike
  __syncthreads();
  constexpr int U = 4;
  for (i64 rb = r0; rb < r1; rb += U * TT) {
    i64 st[U];
    int ln[U], sv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const i64 r = rb + u * TT + tid;
      const bool on = r < r1;
      st[u] = on ? __ldg(R.run_start + r) : 0;
      ln[u] = on ? __ldg(R.run_len + r) : 0;
      sv[u] = on ? __ldg(R.run_s + r) : 0;
    }
    if (R.run_flow && first) {
#pragma unroll
      for (int u = 0; u < U; ++u) { const i64 r = rb + u * TT + tid; if (r < r1) flow += __ldg(R.run_flow + r); }
    }
    if (first) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (ln[u] <= 0) continue;
        if (st[u] < 0) { flags |= 1; continue; }
        const i64 end = st[u] + ln[u];
        steps += ln[u];
        hmax = max_i64(hmax, end);
        flags |= (end > cap ? 2 : 0) | (sv[u] < 0 ? 4 : 0);
        total += static_cast<u64>(static_cast<i64>(sv[u]) + ln[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (ln[u] <= 0 || st[u] < 0) continue;
      const i64 rs = st[u] - t0, re = rs + ln[u];          // from the tile's first round on
      if (re <= 0) continue;
      last = max(last, static_cast<int>(min_i64(re, tile)));
      if (rs >= tile) continue;
      const u32 c = static_cast<u32>(sv[u]) + 1u - static_cast<u32>(st[u]);
      if (rs < 0) { A0 += c; B0 += 1u; }
      else { atomicAdd(&dA[rs], c); atomicAdd(&dB[rs], 1u); }
      if (re < tile) { atomicAdd(&dA[re], 0u - c); atomicAdd(&dB[re], 0xffffffffu); }
    }
  }
  if (first) {
    hmax = block_max(hmax, red64, static_cast<i64>(0));
    total = block_sum(total, redu);
    flags = block_max(flags & 1, red32, 0) | block_max(flags & 2, red32, 0) | block_max(flags & 4, red32, 0);
    if ((flags & 4) || total >= (static_cast<u64>(1) << 32)) {
      // the 64-bit kernel, which runs next, writes every output of this evaluation, also those that its other tiles have written
      if (tid == 0) p.wide_list[atomicAdd(p.wide_count, 1u)] = e;
      return;
    }
  }
  last = block_max(last, red32, 0);
  A0 = block_sum(A0, scanA);
  B0 = block_sum(B0, scanB);
  if (first) {
    steps = block_sum(steps, red64);
    flow = block_sum(flow, red64);
  }
  // prefix sums over the tile: a thread's stretch, then the threads
  const i64 t_end = min_i64(t0 + last, cap);              // rounds [t0, t_end) of this tile exist
  const int e0 = tid * per;
  u32 sa = 0, sb = 0;
  for (int i = 0; i < per; ++i) { sa += dA[e0 + i]; sb += dB[e0 + i]; }
  u32 ia = sa, ib = sb;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const u32 ya = __shfl_up_sync(0xffffffffu, ia, d), yb = __shfl_up_sync(0xffffffffu, ib, d);
    if (lane >= d) { ia += ya; ib += yb; }
  }
  __syncthreads();
  if (lane == 31) { scanA[warp] = ia; scanB[warp] = ib; }
  __syncthreads();
  u32 A = A0 + ia - sa, B = B0 + ib - sb;
  for (int w = 0; w < warp; ++w) { A += scanA[w]; B += scanB[w]; }
  u32 peak = 0;
  const u32 tb = static_cast<u32>(t0) + static_cast<u32>(e0);
  const i64 room = t_end - t0 - e0;                       // rounds of the stretch that exist
  for (int i = 0; i < per; ++i) {
    A += dA[e0 + i]; B += dB[e0 + i];
    const u32 mem = A + (tb + static_cast<u32>(i)) * B;
    if (i < room) peak = max(peak, mem);
    dA[e0 + i] = mem;
  }
  __syncthreads();
  if (p.ev.profile) {
    int32_t* const dst = p.ev.profile + pbase + t0;
    const i64 n = t_end - t0;
    for (i64 i = tid; i < n; i += TT) { const u32 m = dA[i]; __stcs(dst + i, static_cast<int32_t>(m > 0x7fffffffu ? 0x7fffffffu : m)); }
    if (p.fill) block_fill(p.ev.profile + pbase, max_i64(t_end, t0), min_i64(cap, t1), p.fill_prof);
  }
  peak = block_max(peak, scanA, 0u);
  if (tid != 0) return;
  // the tile that finishes last holds the largest memory of all of them
  atomicMax(&p.tile_peak[e], peak);
  if (first) {
    if (p.ev.flow) p.ev.flow[e] = flow;
    if (p.ev.job_steps) p.ev.job_steps[e] = steps;
    if (p.ev.horizon) p.ev.horizon[e] = hmax;
  }
  __threadfence();
  // finished tiles in the lower 28 bits, the first tile's flags above them
  const u32 mine = first ? 1u + (static_cast<u32>(flags) << 28) : 1u, sum = atomicAdd(&p.tile_done[e], mine) + mine;
  if ((sum & 0x0fffffffu) != static_cast<u32>(n_tiles)) return;
  const bool bad = (sum >> 28 & 1u) != 0, clipped = (sum >> 29 & 1u) != 0;
  __threadfence();
  const i64 top = static_cast<i64>(atomicMax(&p.tile_peak[e], 0u));
  int status = 0;
  if (bad) status |= KVS_EVAL_BAD_INPUT;
  if (clipped) status |= KVS_EVAL_CAPACITY;
  if (top > 0x7fffffffll && p.ev.profile) status |= KVS_EVAL_RANGE;
  if (p.ev.peak) p.ev.peak[e] = top;
  if (p.ev.feasible) p.ev.feasible[e] = (!bad && !clipped && R.M && top <= R.M[e]) ? 1 : 0;
  if (p.ev.status) p.ev.status[e] = status;
}

// ---- one CTA per evaluation, arrays in global memory, 64-bit arithmetic ---------------------------------

__global__ void __launch_bounds__(T) k_generic_eval(GenericParams p) {
  __shared__ i64 red64[32];
  __shared__ int red32[32];
  __shared__ i64 scanA[32];
  __shared__ int scanB[32];
  const int tid = threadIdx.x;
  const kvs_runs& R = p.runs;
  const bool listed = p.wide_list && !*p.odd;
  const i64 n_list = listed ? static_cast<i64>(*p.wide_count) : R.P;
  for (i64 at = blockIdx.x; at < n_list; at += gridDim.x) {
    const i64 e = listed ? p.wide_list[at] : at;
    const i64 r0 = R.run_off[e], r1 = R.run_off[e + 1];
    const i64 pbase = p.ev.profile_off[e];
    const i64 cap = p.ev.profile_off[e + 1] - pbase;
    // The difference arrays hold `slots` entries; evaluation e owns entries pbase + e .. pbase + e + cap.
    // Offsets on the device that do not fit (not monotone, or larger than the host said when the arrays
    // were sized) would send the atomics outside them: such an evaluation is reported and skipped.
    if (pbase < 0 || cap < 0 || pbase > p.slots || cap > p.slots - pbase || e + 1 > p.slots - pbase - cap) {
      if (tid == 0) {
        if (p.ev.peak) p.ev.peak[e] = -1;
        if (p.ev.flow) p.ev.flow[e] = 0;
        if (p.ev.job_steps) p.ev.job_steps[e] = 0;
        if (p.ev.horizon) p.ev.horizon[e] = 0;
        if (p.ev.feasible) p.ev.feasible[e] = 0;
        if (p.ev.status) p.ev.status[e] = KVS_EVAL_CAPACITY | KVS_EVAL_BAD_INPUT;
      }
      continue;
    }
    i64* const dA = p.dconst + pbase + e;      // cap + 1 entries
    int32_t* const dB = p.dcount + pbase + e;
    if (p.wide_list) {                        // the caller has cleared nothing for a list
      for (i64 i = tid; i <= cap; i += T) { dA[i] = 0; dB[i] = 0; }
      __threadfence();
      __syncthreads();
    }
    i64 steps = 0, hmax = 0, flow = 0;
    int bad = 0, clipped = 0;
    for (i64 r = r0 + tid; r < r1; r += T) {
      const i64 start = R.run_start[r];
      const i64 len = R.run_len[r];
      if (R.run_flow) flow += R.run_flow[r];
      if (len <= 0) continue;
      if (start < 0) { bad = 1; continue; }
      const i64 end = start + len;
      steps += len;
      hmax = max_i64(hmax, end);
      const i64 c = static_cast<i64>(R.run_s[r]) + 1 - start;
      if (end > cap) clipped = 1;
      if (start < cap) {
        atomicAdd(reinterpret_cast<ull*>(dA + start), static_cast<ull>(c));
        atomicAdd(dB + start, 1);
        if (end <= cap) {
          atomicAdd(reinterpret_cast<ull*>(dA + end), static_cast<ull>(-c));
          atomicAdd(dB + end, -1);
        }
      }
    }
    steps = block_sum(steps, red64);
    hmax = block_max(hmax, red64, static_cast<i64>(0));
    flow = block_sum(flow, red64);
    bad = block_max(bad, red32, 0);
    clipped = block_max(clipped, red32, 0);
    __threadfence();
    __syncthreads();

    const i64 t_end = hmax < cap ? hmax : cap;
    i64 A_run = 0, peak = 0;
    int B_run = 0, over = 0;
    for (i64 t0 = 0; t0 < t_end; t0 += T * ITEMS) {
      i64 a[ITEMS];
      int b[ITEMS];
      i64 sa = 0;
      int sb = 0;
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const i64 t = t0 + tid * ITEMS + i;
        if (t < t_end) { sa += dA[t]; sb += dB[t]; }
        a[i] = sa; b[i] = sb;
      }
      i64 ia = sa;
      int ib = sb;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const i64 ya = __shfl_up_sync(0xffffffffu, ia, d);
        const int yb = __shfl_up_sync(0xffffffffu, ib, d);
        if (static_cast<int>(lane_id()) >= d) { ia += ya; ib += yb; }
      }
      __syncthreads();
      if (lane_id() == 31) { scanA[tid >> 5] = ia; scanB[tid >> 5] = ib; }
      __syncthreads();
      i64 wa = (lane_id() < T / 32) ? scanA[lane_id()] : 0;
      int wb = (lane_id() < T / 32) ? scanB[lane_id()] : 0;
      i64 wia = wa;
      int wib = wb;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const i64 ya = __shfl_up_sync(0xffffffffu, wia, d);
        const int yb = __shfl_up_sync(0xffffffffu, wib, d);
        if (static_cast<int>(lane_id()) >= d) { wia += ya; wib += yb; }
      }
      const i64 offA = A_run + __shfl_sync(0xffffffffu, wia - wa, tid >> 5) + (ia - sa);
      const int offB = B_run + __shfl_sync(0xffffffffu, wib - wb, tid >> 5) + (ib - sb);
      A_run += __shfl_sync(0xffffffffu, wia, 31);
      B_run += __shfl_sync(0xffffffffu, wib, 31);
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const i64 t = t0 + tid * ITEMS + i;
        if (t < t_end) {
          const i64 mem = (offA + a[i]) + t * static_cast<i64>(offB + b[i]);
          peak = max_i64(peak, mem);
          if (mem > 0x7fffffffll) over = 1;
          if (p.ev.profile) p.ev.profile[pbase + t] = static_cast<int32_t>(mem > 0x7fffffffll ? 0x7fffffffll : mem);
        }
      }
    }
    if (p.fill && p.ev.profile) block_fill(p.ev.profile + pbase, t_end, cap, p.fill_prof);
    peak = block_max(peak, red64, static_cast<i64>(0));
    over = block_max(over, red32, 0);
    if (tid == 0) {
      int status = 0;
      if (bad) status |= KVS_EVAL_BAD_INPUT;
      if (clipped) status |= KVS_EVAL_CAPACITY;
      if (over && p.ev.profile) status |= KVS_EVAL_RANGE;
      if (p.ev.peak) p.ev.peak[e] = peak;
      if (p.ev.flow) p.ev.flow[e] = flow;
      if (p.ev.job_steps) p.ev.job_steps[e] = steps;
      if (p.ev.horizon) p.ev.horizon[e] = hmax;
      if (p.ev.feasible) p.ev.feasible[e] = (!bad && !clipped && R.M && peak <= R.M[e]) ? 1 : 0;
      if (p.ev.status) p.ev.status[e] = status;
    }
    __syncthreads();
  }
}

}  // namespace

// Once per device, before the first launch.
cudaError_t kvs_setup_generic() {
  return cudaFuncSetAttribute(k_tile_eval, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * TILE_MAX * 4);
}

// The tiled kernel over capacity_total rounds, then what it has listed.  Tiles are as large as shared memory allows with two
// CTAs per SM; fewer evaluations than that fills get smaller tiles (every tile reads all runs of its evaluation, so
// no more tiles than it takes to give every SM two).
cudaError_t kvs_launch_generic_tiled(GenericParams p, i64 capacity_total, int sm_count, cudaStream_t stream) {
  if (p.runs.P <= 0) return cudaSuccess;
  i64 per = capacity_total / (2ll * sm_count) / TT;
  per = per < 3 ? 3 : (per > TK ? TK : per | 1);
  p.tile = per * TT;
  const i64 items = capacity_total / p.tile + p.runs.P;
  if (items >= (static_cast<i64>(1) << 31)) return cudaErrorInvalidConfiguration;
  k_tile_init<<<static_cast<unsigned>((p.runs.P + 255) / 256), 256, 0, stream>>>(p, capacity_total);
  k_tile_eval<<<static_cast<unsigned>(items), TT, static_cast<size_t>(2 * p.tile * 4), stream>>>(p);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int grid = static_cast<int>(p.runs.P < 2 * sm_count ? p.runs.P : 2 * sm_count);
  k_generic_eval<<<grid, T, 0, stream>>>(p);
  return cudaGetLastError();
}

cudaError_t kvs_launch_generic(const GenericParams& p, cudaStream_t stream) {
  if (p.runs.P <= 0) return cudaSuccess;
  const int grid = static_cast<int>(p.runs.P < 4096 ? p.runs.P : 4096);
  k_generic_eval<<<grid, T, 0, stream>>>(p);
  return cudaGetLastError();
}

// ---- variant without any caller- or library-allocated scratch -----------------------------------
//
// Same kernel, but the two difference arrays live in a fixed array that is part of the loaded
// library image on every GPU (12 MiB per device, held until the process exits).  The array is
// shared by all calls on a device and keeps what the previous call left, so each call clears the
// part it uses first; two calls that overlap on the GPU would race on it.

constexpr int64_t KVS_NOALLOC_SLOTS = int64_t(1) << 20;   // rounds + evaluations per call
static __device__ __align__(256) unsigned char kvs_noalloc_scratch[KVS_NOALLOC_SLOTS * 12];

namespace {
constexpr int KVS_NOALLOC_MAX_DEVICES = 64;
// Device address of the array, per device.  Atomic, so that two host threads making their first call on
// a device at the same time both end up with the same, fully written pointer.
std::atomic<void*> g_noalloc_ptr[KVS_NOALLOC_MAX_DEVICES] = {};
void put_msg(char* err, uint64_t len, const char* msg) {
  if (err && len) { snprintf(err, static_cast<size_t>(len), "%s", msg); }
}
}  // namespace

extern "C" int kvs_evaluate_schedule_noalloc(int32_t device, void* stream, const kvs_runs* runs,
                                             const kvs_eval_out* ev, int64_t capacity_total,
                                             char* err, uint64_t err_len) {
  if (!runs || !ev) { put_msg(err, err_len, "runs or eval_out is null"); return KVS_E_ARG; }
  if (runs->P < 0 || capacity_total < 0) { put_msg(err, err_len, "negative size"); return KVS_E_ARG; }
  if (device < 0 || device >= KVS_NOALLOC_MAX_DEVICES) { put_msg(err, err_len, "device ordinal out of range"); return KVS_E_ARG; }
  if (runs->P == 0) return KVS_OK;
  if (!runs->run_off || !runs->run_start || !runs->run_len || !runs->run_s || !ev->profile_off) {
    put_msg(err, err_len, "null run array or profile_off");
    return KVS_E_ARG;
  }
  if (runs->P > KVS_NOALLOC_SLOTS || capacity_total > KVS_NOALLOC_SLOTS - runs->P) {
    put_msg(err, err_len, "capacity_total + P exceeds the 1,048,576 slots of the built-in scratch array; "
                          "use kvs_evaluate_schedule with a workspace instead");
    return KVS_E_CAPACITY;
  }
  // The work is issued with `device` current; the caller's current device is put back before returning.
  int prev_device = -1;
  cudaError_t ce = cudaGetDevice(&prev_device);
  if (ce == cudaSuccess && prev_device != device) ce = cudaSetDevice(device);
  if (ce != cudaSuccess) { put_msg(err, err_len, cudaGetErrorString(ce)); return KVS_E_CUDA; }
  struct Restore {
    int prev, cur;
    ~Restore() { if (prev >= 0 && prev != cur) cudaSetDevice(prev); }
  } restore{prev_device, device};
  void* ptr = g_noalloc_ptr[device].load(std::memory_order_acquire);
  if (!ptr) {
    // In host code the array's name is only a handle; its device address has to be asked for,
    // once per device, with that device current.
    ce = cudaGetSymbolAddress(&ptr, kvs_noalloc_scratch);
    if (ce != cudaSuccess || !ptr) { put_msg(err, err_len, cudaGetErrorString(ce)); return KVS_E_CUDA; }
    g_noalloc_ptr[device].store(ptr, std::memory_order_release);
  }
  unsigned char* base = static_cast<unsigned char*>(ptr);
  const size_t slots = static_cast<size_t>(capacity_total + runs->P);
  const size_t bytes_a = (slots * 8 + 255) & ~static_cast<size_t>(255);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  ce = cudaMemsetAsync(base, 0, bytes_a + slots * 4, s);   // what must start at zero
  if (ce != cudaSuccess) { put_msg(err, err_len, cudaGetErrorString(ce)); return KVS_E_CUDA; }
  GenericParams gp{};
  gp.runs = *runs;
  gp.ev = *ev;
  gp.dconst = reinterpret_cast<i64*>(base);
  gp.dcount = reinterpret_cast<int32_t*>(base + bytes_a);
  gp.slots = static_cast<i64>(slots);
  ce = kvs_launch_generic(gp, s);
  if (ce != cudaSuccess) { put_msg(err, err_len, cudaGetErrorString(ce)); return KVS_E_CUDA; }
  return KVS_OK;
}
