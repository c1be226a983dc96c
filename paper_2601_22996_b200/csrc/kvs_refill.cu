// Dynamic refill of batching schedules (Numerical Experiments, "Dynamic Refill (GBA-D)"): a job is admitted
// as soon as the pipeline can go on with it without violating memory feasibility, no job is delayed relative
// to the batching schedule, only idle time is filled.
//
// The rule is sequential - every admission changes the memory the next one sees - so one CTA works on one evaluation and
// many evaluations run side by side.  It starts from what the fused kernels left: every job's start in the batching schedule
// and the per-round memory of that schedule (the plan).  Jobs are taken in the schedule's order (key order).  A job's ramp
// s + u + 1 is taken out of the plan, the earliest round t between the previous admission and the job's old start is
// found at which the ramp fits on top of the plan in every round, and the ramp is put back there.  With R(u) = plan(u) + u
// the ramp fits from t on iff max over u in [t, t + o) of R(u) <= M - s - 1 + t; if it does not, the maximising round
// u* rules out every start before min(max R - (M - s - 1), u* + 1), so the search jumps there instead of trying round by round.
//
// What bounds it is the chain of dependent reads per job, so the rounds that a job can touch are kept in shared memory.
// Admissions are monotone and the old starts too, hence a job looks at the rounds [t, t + o) from the previous
// admission on, and the response lengths grow along the order: a ring of RING rounds from the last admission holds
// everything until the first job with o > RING (a handful per instance; from there on the whole CTA works on the plan in
// global memory).  A round that enters the ring holds what the batching schedule has there less the ramps of the jobs
// already taken: nothing before the next job's old start, otherwise the stored profile minus the few of those
// ramps that reach so far (old starts therefore stay in job_start until the end; the new ones wait in job_completion).
// One warp walks the ring; the next 32 to 64 jobs are loaded ahead, and up to 32 of them, of about the same length, are tried together.
// A call of 1,024 evaluations of 5,000 to 10,000 jobs, batching schedules included: 3.0 ms (jobs of one length together, eight at a time,
// every one of the eight tested, and 128 threads with four loads in flight for the long ones: 4.3; one warp per evaluation on the
// plan in global memory: 21).
#include "kvs_check.cuh"

namespace {

constexpr int RT = 128;
constexpr int RING = 4096;              // 16 KB
constexpr int FILL = 128;               // rounds that enter the ring together

struct Job { int j, o, s, g; };

// One warp hides no latency by itself, so what it costs is the number of instructions in a row: the ring is
// read and written four rounds per lane at a time.  quads<WRITE>(ring, u0, u1, f): f(rel, word) for the rounds u0 + rel < u1, the
// returned word is stored if WRITE (words of a quad outside the range are stored as they were).
template <bool WRITE, class F>
__device__ __forceinline__ void quads(int* ring, int u0, int u1, F f) {
  const u32 len = static_cast<u32>(u1 - u0);
  for (int q = (u0 & ~3) + 4 * static_cast<int>(lane_id()); q < u1; q += 128) {
    int4* const at = reinterpret_cast<int4*>(ring + (q & (RING - 1)));
    int4 v = *at;
    const int rel = q - u0;
    if (static_cast<u32>(rel) < len) v.x = f(rel, v.x);
    if (static_cast<u32>(rel + 1) < len) v.y = f(rel + 1, v.y);
    if (static_cast<u32>(rel + 2) < len) v.z = f(rel + 2, v.z);
    if (static_cast<u32>(rel + 3) < len) v.w = f(rel + 3, v.w);
    if (WRITE) *at = v;
  }
}

__global__ void __launch_bounds__(RT) k_refill(RefillParams p) {
  __shared__ alignas(16) int ring[RING];
  __shared__ int4 sh_job[64];
  __shared__ int sh_next, sh_prev, sh_filled, sh_max[32];
  __shared__ i64 sh_best[RT / 32], sh_peak[32];
  __shared__ int sh_arg[RT / 32];
  __shared__ i64 sh_sum[32];
  const int lane = lane_id(), tid = threadIdx.x;
  const i64 e = p.eval_list[blockIdx.x];
  if (p.status && p.status[e] != 0) return;            // the batching schedule was not formed or not stored in full
  const kvs_setting st = p.settings[e];
  const i64 lo = p.job_off[st.instance];
  const int n = static_cast<int>(p.job_off[st.instance + 1] - lo);
  const i64 M = st.M;
  int32_t* const prof = p.profile + p.profile_off[e];
  int32_t* const js = p.job_start + p.job_out_off[e];
  int32_t* const jc = p.job_completion + p.job_out_off[e];
  const int32_t* const perm = p.perm + lo;
  const int32_t* const So = p.sorted_s + lo;
  const int32_t* const Oo = p.sorted_o + lo;
  const int H = static_cast<int>(p.horizon[e]);         // of the batching schedule; within the profile's capacity (status 0)
  const i64 pcap = p.profile_off[e + 1] - p.profile_off[e];   // bound of every profile index below (checked build)
  (void)pcap;
  auto load = [&](int x) {
    Job b{0, 0x7fffffff, 0, 0x7fffffff};
    if (x < n) {
      b.j = perm[x]; b.o = Oo[x]; b.s = So[x];
      if (!KVS_OK_AT(b.j, n, CHK_RF_JOB)) b.j = 0;
      b.g = js[b.j];
    }
    return b;
  };
  // Takes the old ramps of the jobs before `x` out of rounds [v0, v1) of the stored profile, by one warp; ring: of the ring.
  auto take_out = [&](int x, int v0, int v1, int o_last, bool in_ring) {
    for (int y = x - 1; y >= 0; y -= 32) {
      const int z = y - lane;
      Job b{0, 0, 0, 0};
      if (z >= 0) b = load(z);
      // old starts and response lengths grow along the order: nothing further back reaches v0 once this holds
      const int g_top = __shfl_sync(0xffffffffu, b.g, 0);
      if (static_cast<i64>(g_top) + o_last <= v0) break;
      u32 m = __ballot_sync(0xffffffffu, z >= 0 && b.g < v1 && b.g + b.o > v0);
      while (m) {
        const int src = __ffs(static_cast<int>(m)) - 1;
        m &= m - 1u;
        const int g = __shfl_sync(0xffffffffu, b.g, src), o = __shfl_sync(0xffffffffu, b.o, src), s = __shfl_sync(0xffffffffu, b.s, src);
        const int u1 = min(g + o, v1);
        for (int u = max(g, v0) + lane; u < u1; u += 32) {
          if (in_ring) ring[u & (RING - 1)] -= s + (u - g) + 1;
          else if (KVS_OK_AT(u, pcap, CHK_RF_PROF_OUT)) prof[u] -= s + (u - g) + 1;
        }
        __syncwarp();
      }
    }
  };

  if (tid < 32) {
    int base = 0, filled = 0;                           // the ring holds rounds [base, filled)
    int x0 = 0;
    bool tail = false;
    bool negative = false;                              // a word of the plan does not fit 31 bits: no short cuts
    // No admission before round t any more: the rounds before it are final.
    auto advance = [&](int t) {
      for (int u = base + lane; u < t; u += 32)
        if (KVS_OK_AT(u, pcap, CHK_RF_PROF_OUT)) __stcs(prof + u, ring[u & (RING - 1)]);
      __syncwarp();
      base = t;                                         // at most the last window's end, so within the filled rounds
    };
    // Rounds up to `need` enter the ring: without the old ramps of the jobs before y, the next of which starts at g_y.
    auto fill_to = [&](int y, int need, int g_y, int o_last) {
      const int v1 = min(max(filled + FILL, need), base + RING - 4);
      const bool nothing = v1 <= g_y;
      bool neg = false;
      for (int u = filled + lane; u < v1; u += 32) {
        const int v = (nothing || u >= H || !KVS_OK_AT(u, pcap, CHK_RF_PROF_WIN)) ? 0 : prof[u];
        neg |= v < 0;
        ring[u & (RING - 1)] = v;
      }
      __syncwarp();
      negative |= __any_sync(0xffffffffu, neg) != 0;
      if (!nothing) take_out(y, filled, v1, o_last, true);
      filled = v1;
    };
    // Memory modulo 2^32: a word of the plan is below 2^31, the prompts of `most_jobs` jobs that fit M one by one are below 2^32, and
    // 2^20 is room for the slopes of 32 jobs over the ring.
    const u32 Mu = static_cast<u32>(M);
    const int most_jobs = M >> 27 ? static_cast<int>(0xffffffffu / Mu) : 32;
    if (M > (1ll << 31) - (1 << 20)) negative = true;
    // jobs x0 .. x0 + 63 lie in sh_job (job x at x mod 64: response, sum of s + 1 up to it modulo 2^32, old start, index), the 32 after
    // them are on their way
    u32 sum = 0;
    auto keep = [&](int from, const Job& b) {
      const u32 P = sum + warp_incl(static_cast<u32>(b.s) + 1u);
      sh_job[(from + lane) & 63] = make_int4(b.o, static_cast<int>(P), b.g, b.j);
      sum = __shfl_sync(0xffffffffu, P, 31);
    };
    u32 before = 0;                                     // the sum up to the job before x
    keep(0, load(lane));
    Job nxt = load(32 + lane);
    int x = 0;
    for (; x0 < n && !tail; x0 += 32) {
      keep(x0 + 32, nxt);
      __syncwarp();
      nxt = load(x0 + 64 + lane);
      const int m = min(32, n - x0);
      while (x < m) {
        const int4 b = sh_job[(x0 + x) & 63], c = sh_job[(x0 + x + lane) & 63];   // the next job; lane i: the i-th from here on
        const int o = b.x, g = b.z;
        if (o > RING - 4) { tail = true; break; }
        const int t = base;
        // the jobs that may be tried together, see below
        const u32 near = __ballot_sync(0xffffffffu, c.x <= min(min(o + (o >> 3) + 32, RING - 4), g - t));
        const int cnt = min(most_jobs, near == 0xffffffffu ? 32 : __ffs(static_cast<int>(~near)) - 1);
        const bool alone = cnt == 0;
        const int o_last = __shfl_sync(0xffffffffu, c.x, max(cnt - 1, 0));
        if (filled < t + o_last) fill_to(x0 + x, t + o_last, g, o_last);
        if (g <= t) {                                   // its turn comes at its old start: it stays where it is
          if (lane == 0) jc[b.w] = g + o;
          before = static_cast<u32>(b.y);
          ++x;
          continue;
        }
        if (!negative) {
          // Most jobs fit where the last one was admitted, and neighbours in the order have about the same response lengths: up to
          // 32 of them are tried together there, if their old ramps (and so those of all later jobs) begin behind their windows.
          // With N the plan, the first k fit if N(t + r) + S_k + k r <= M for every r below the k-th's length, S_k the sum of
          // their s + 1 (exactly then, if their lengths are equal; otherwise the shorter ones are counted beyond their ends, and
          // those that do not fit so are tried again behind the others).  Memory only grows with k, so many that fit are
          // found by testing one k, cutting it down to what the worst round leaves, and so on; for k = 1 the test is exact.
          // A job whose old ramp begins inside its window, G rounds behind t, is tried alone: there the plan loses the old
          // ramp and gets the new one, which is G more.
          const int q0 = t & ~3;
          const u32 G = static_cast<u32>(g - t);
          const u32 S = static_cast<u32>(c.y) - before;
          // how many jobs round r leaves room for
          auto room_at = [&](u32 r) {
            const u32 used = static_cast<u32>(ring[(t + static_cast<int>(r)) & (RING - 1)]) + static_cast<u32>(lane + 1) * r;
            return __popc(__ballot_sync(0xffffffffu, lane < cnt && used <= Mu && S <= Mu - used));
          };
          const bool once = q0 + 256 >= t + o_last;                    // one step covers the window: its words are read once
          u32 A, C, len, w[8];
          // the eight words of this lane from round q on
          auto read = [&](int q) {
            const int4 v0 = *reinterpret_cast<const int4*>(ring + (q & (RING - 1)));
            const int4 v1 = *reinterpret_cast<const int4*>(ring + ((q + 128) & (RING - 1)));
            w[0] = v0.x; w[1] = v0.y; w[2] = v0.z; w[3] = v0.w; w[4] = v1.x; w[5] = v1.y; w[6] = v1.z; w[7] = v1.w;
          };
          // f(i, r, what the jobs tried add there) for those of them that lie in the window
          auto each = [&](int q, auto f) {
            const u32 r0 = static_cast<u32>(q - t), a0 = A + C * r0;
            if (!alone) {
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const u32 d = static_cast<u32>(i < 4 ? i : 124 + i);
                if (r0 + d < len) f(i, r0 + d, a0 + C * d);
              }
            } else {
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const u32 d = static_cast<u32>(i < 4 ? i : 124 + i);
                if (r0 + d < len) f(i, r0 + d, r0 + d < G ? a0 + d : G);
              }
            }
          };
          if (once) read(q0 + 4 * lane);
          int k = alone ? 1 : max(1, min(room_at(0u), room_at(static_cast<u32>(o) - 1u)));
          u32 most, arg = 0;                                           // the worst round and the memory in it
          for (;;) {
            A = __shfl_sync(0xffffffffu, S, k - 1);
            C = static_cast<u32>(k);
            len = static_cast<u32>(__shfl_sync(0xffffffffu, c.x, k - 1));
            const int end = t + static_cast<int>(len);
            u32 top = 0, at = 0;
            int q_top = q0 + 4 * lane;
            for (int q = q0 + 4 * lane; q - 4 * lane < end; q += 256) {
              if (!once) read(q);
              u32 here = 0;
              each(q, [&](int i, u32, u32 add) { here = max(here, w[i] + add); });
              if (here >= top) { top = here; q_top = q; }
            }
            most = __reduce_max_sync(0xffffffffu, top);
            if (most <= Mu) break;
            if (!once) read(q_top);
            each(q_top, [&](int i, u32 r, u32 add) { at = w[i] + add == most ? r : at; });
            arg = __reduce_max_sync(0xffffffffu, at);
            if (k == 1) { k = 0; break; }
            k = room_at(arg);
            if (k == 0) {
              if (arg >= static_cast<u32>(o)) { k = 1; continue; }     // behind the first one's window
              most = static_cast<u32>(ring[(t + static_cast<int>(arg)) & (RING - 1)]) + __shfl_sync(0xffffffffu, S, 0) + arg;
              break;
            }
          }
          if (k > 0) {
            const u32 longest = len;
            len = static_cast<u32>(o);                  // all k of them run for so long
            for (int q = q0 + 4 * lane; q - 4 * lane < t + o; q += 256) {
              if (!once) read(q);
              each(q, [&](int i, u32, u32 add) { w[i] += add; });
              *reinterpret_cast<int4*>(ring + (q & (RING - 1))) = make_int4(w[0], w[1], w[2], w[3]);
              *reinterpret_cast<int4*>(ring + ((q + 128) & (RING - 1))) = make_int4(w[4], w[5], w[6], w[7]);
            }
            __syncwarp();
            for (u32 r0 = len; r0 < longest; r0 += 32) {  // then one after the other ends
              const u32 r = r0 + lane;
              int ended = 0;                            // of the first k, in order
#pragma unroll
              for (int d = 16; d > 0; d >>= 1) {
                const int v = __shfl_sync(0xffffffffu, c.x, ended + d - 1);
                if (ended + d < k && static_cast<u32>(v) <= r) ended += d;
              }
              const u32 gone = __shfl_sync(0xffffffffu, S, max(ended - 1, 0));
              if (r < longest) ring[(t + static_cast<int>(r)) & (RING - 1)] += static_cast<int>(A - (ended ? gone : 0u) + (C - static_cast<u32>(ended)) * r);
            }
            if (lane < k) jc[c.w] = t + c.x;
            __syncwarp();
            // old ramps that are in the ring leave it
            if (alone) {
              const int first = static_cast<int>(A) - g;
              for (int u = t + o + lane; u < min(g + o, filled); u += 32) ring[u & (RING - 1)] -= first + u;
              __syncwarp();
            } else if (g < filled) {
              u32 in = __ballot_sync(0xffffffffu, lane < k && c.z < filled);
              const u32 left_of = __shfl_up_sync(0xffffffffu, S, 1), s1 = lane > 0 ? S - left_of : S;
              while (in) {
                const int src = __ffs(static_cast<int>(in)) - 1;
                in &= in - 1u;
                const int gs = __shfl_sync(0xffffffffu, c.z, src), os = __shfl_sync(0xffffffffu, c.x, src);
                const int first = static_cast<int>(__shfl_sync(0xffffffffu, s1, src));
                quads<true>(ring, gs, min(gs + os, filled), [&](int rel, int v) { return v - (first + rel); });
                __syncwarp();
              }
            }
            x += k;
            before += A;
          } else {
            // no start before that round has passed, or before the plan may be that high
            advance(static_cast<int>(min_i64(t + min_i64(static_cast<i64>(most) - M, static_cast<i64>(arg) + 1), static_cast<i64>(g))));
          }
          continue;
        }
        // One job on a plan with words beyond 31 bits: its old ramp leaves the ring first.
        const int s = static_cast<int>(static_cast<u32>(b.y) - before - 1u), j = b.w, g_next = sh_job[(x0 + x + 1) & 63].z;
        if (g < filled) {
          quads<true>(ring, g, min(g + o, filled), [&](int rel, int v) { return v - (s + rel + 1); });
          __syncwarp();
        }
        const i64 bound = M - s - 1;
        int d = g;
        for (;;) {
          if (filled < base + o) fill_to(x0 + x + 1, base + o, g_next, o);
          const int t = base;
          if (t >= g) break;
          // max of plan(u) + u over the window, and the last round that attains it
          i64 best = -1;
          int arg = t;
          quads<false>(ring, t, t + o, [&](int rel, int v) {
            const i64 y = static_cast<i64>(v) + t + rel;
            if (y >= best) { best = y; arg = t + rel; }
            return 0;
          });
          if (!__any_sync(0xffffffffu, best - t > bound)) { d = t; break; }
#pragma unroll
          for (int dd = 16; dd > 0; dd >>= 1) {
            const i64 ob = __shfl_xor_sync(0xffffffffu, best, dd);
            const int oa = __shfl_xor_sync(0xffffffffu, arg, dd);
            if (ob > best || (ob == best && oa > arg)) { best = ob; arg = oa; }
          }
          advance(static_cast<int>(min_i64(min_i64(best - bound, static_cast<i64>(arg) + 1), static_cast<i64>(g))));
        }
        quads<true>(ring, d, d + o, [&](int rel, int v) { return v + s + rel + 1; });
        __syncwarp();
        if (lane == 0) jc[j] = d + o;
        before = static_cast<u32>(b.y);
        ++x;
      }
      if (tail) { x0 += x; break; }
      x -= 32;                                          // jobs of the next 32 that have been taken already
    }
    x0 = min(x0, n);
    if (lane == 0) { sh_next = x0; sh_prev = base; sh_filled = filled; }
  }
  __syncthreads();
  // the ring goes back to the plan, the rest of which holds the remaining jobs' old ramps only
  const int next = sh_next, filled = sh_filled;
  const bool tail = next < n;
  const int j_next = tail ? perm[next] : 0;
  const int g_next = tail && KVS_OK_AT(j_next, n, CHK_RF_JOB) ? js[j_next] : H;
  for (int u = sh_prev + tid; u < min(filled, H); u += RT)
    if (KVS_OK_AT(u, pcap, CHK_RF_PROF_OUT)) prof[u] = ring[u & (RING - 1)];
  for (int u = filled + tid; u < min(g_next, H); u += RT)
    if (KVS_OK_AT(u, pcap, CHK_RF_PROF_OUT)) prof[u] = 0;
  __syncthreads();
  // ---- jobs that are longer than the ring: the whole CTA, the plan in global memory ----
  int prev = sh_prev;
  if (tail) {
    if (tid < 32 && next > 0) take_out(next, max(filled, g_next), H, Oo[next - 1], false);
    __syncthreads();
  }
  constexpr int U = 8;                                  // loads in flight per thread
  for (int x = next; x < n; ++x) {
    const Job b = load(x);
    const int o = b.o, g = b.g;
    const i64 bound = M - b.s - 1;
    int d = g, t = prev;
    // the job's own old ramp stays in the plan until its new start is known: it is left out of what is read
    while (t < g) {
      i64 best = -1;
      int arg = t;
      for (int u0 = t + tid; u0 < t + o; u0 += U * RT) {
        int v[U];
#pragma unroll
        for (int i = 0; i < U; ++i) { const int u = u0 + i * RT; v[i] = u < t + o && KVS_OK_AT(u, pcap, CHK_RF_PROF_WIN) ? prof[u] : -1; }
#pragma unroll
        for (int i = 0; i < U; ++i) {
          const int u = u0 + i * RT;
          const i64 r = static_cast<i64>(v[i] - (u >= g ? b.s + (u - g) + 1 : 0)) + u;
          if (u < t + o && r >= best) { best = r; arg = u; }
        }
      }
#pragma unroll
      for (int dd = 16; dd > 0; dd >>= 1) {
        const i64 ob = __shfl_xor_sync(0xffffffffu, best, dd);
        const int oa = __shfl_xor_sync(0xffffffffu, arg, dd);
        if (ob > best || (ob == best && oa > arg)) { best = ob; arg = oa; }
      }
      if (lane == 0) { sh_best[tid >> 5] = best; sh_arg[tid >> 5] = arg; }
      __syncthreads();
      for (int w = 0; w < RT / 32; ++w)
        if (sh_best[w] > best || (sh_best[w] == best && sh_arg[w] > arg)) { best = sh_best[w]; arg = sh_arg[w]; }
      __syncthreads();
      if (best - t <= bound) { d = t; break; }
      t = static_cast<int>(min_i64(best - bound, static_cast<i64>(arg) + 1));
    }
    if (d < g) {                                        // out at the old start, in at the new one
      auto move = [&](int from, int to) {
        for (int u0 = from + tid; u0 < to; u0 += U * RT) {
          int v[U];
#pragma unroll
          for (int i = 0; i < U; ++i) { const int u = u0 + i * RT; v[i] = u < to && KVS_OK_AT(u, pcap, CHK_RF_PROF_IN) ? prof[u] : 0; }
#pragma unroll
          for (int i = 0; i < U; ++i) {
            const int u = u0 + i * RT;
            if (u < to && KVS_OK_AT(u, pcap, CHK_RF_PROF_OUT)) prof[u] = v[i] + (u < d + o ? b.s + (u - d) + 1 : 0) - (u >= g ? b.s + (u - g) + 1 : 0);
          }
        }
      };
      move(d, min(d + o, g));
      move(g, g + o);
      __syncthreads();
    }
    if (tid == 0) jc[b.j] = d + o;
    prev = d;
  }
  __syncthreads();
  // the starts: completion less response, both by position now; flow and horizon
  i64 flow = 0;
  int hmax = 0;
  for (int x0 = tid; x0 < n; x0 += U * RT) {
    int j[U], v[U];
#pragma unroll
    for (int i = 0; i < U; ++i) { const int x = x0 + i * RT; j[i] = x < n ? perm[x] : 0; v[i] = x < n ? Oo[x] : 0; }
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int end = x0 + i * RT < n && KVS_OK_AT(j[i], n, CHK_RF_JOB) ? jc[j[i]] : 0;
      flow += end;
      hmax = max(hmax, end);
      v[i] = end - v[i];
    }
#pragma unroll
    for (int i = 0; i < U; ++i) if (x0 + i * RT < n && KVS_OK_AT(j[i], n, CHK_RF_JOB)) js[j[i]] = v[i];
  }
  flow = block_sum(flow, sh_sum);
  hmax = block_max(hmax, sh_max, 0);
  int most = 0;
#pragma unroll 8
  for (int u = tid; u < hmax; u += RT) most = max(most, prof[u]);
  i64 peak = most;
  peak = block_max(peak, sh_peak, static_cast<i64>(0));
  if (tid == 0) {
    if (p.peak) p.peak[e] = peak;
    if (p.flow) p.flow[e] = flow;
    p.horizon[e] = hmax;
    if (p.feasible) p.feasible[e] = peak <= M ? 1 : 0;
  }
}

}  // namespace

KVS_DEFINE_CHECK_WORD(kvs_refill_check_word)

cudaError_t kvs_launch_refill(const RefillParams& p, cudaStream_t stream) {
  if (p.n_list <= 0) return cudaSuccess;
  k_refill<<<static_cast<unsigned>(p.n_list), RT, 0, stream>>>(p);
  return cudaGetLastError();
}
