// Speculative runs on top of slicing schedules (Numerical Experiments, "Speculative Runs (GSA-Spec)"): memory
// that the pipeline leaves free runs unfinished jobs ahead of their turn; such runs are killed when the
// pipeline needs the memory, so the slicing schedule itself is kept; they start and are killed first come
// first served.
//
// The rule is a round-by-round simulation in which every decision depends on the rounds before it, so one
// warp simulates one evaluation and many evaluations run side by side.  The warp starts from what the fused
// kernels left - the per-round memory of the slicing schedule (the plan) in the caller's profile buffer -
// and forms the pipeline's runs again from the phase table: the participants of phase p are the jobs of class
// p or later in index order, rank r starts at base_p + floor(r tau_p / k_p) and holds its slot for tau_p rounds
// (Procedure StaggeredPipelineSchedule).  Round t:
//   (1) a speculative run that has received all its rounds completes its job;
//   (2) the pipeline's runs that start at t begin: a job that has completed is dropped from the plan (its ramp
//       is taken out of the profile), a job that is running speculatively loses that run;
//   (3) while pipeline and speculative runs together exceed M, the speculative run started last is killed;
//   (4) the jobs that are not done and not running are taken in index order: the lowest one starts a
//       speculative run if its first round fits (s + 1 tokens), then the next, until one does not fit;
//   (5) the round's memory, pipeline + speculative, is written over the plan's entry.
// The speculative runs hold A + t * count tokens in round t (a run started at t0 holds s + 1 - t0 + t).
// Per phase the participants are kept as a list in index order, so that rank r is entry r.  Two cursors walk
// it: one over the run starts, one over the slot ends start + tau (nondecreasing in the rank), which is when a
// killed job becomes free to speculate.  No entry before position `fpos` and none at or after `fhi` is free at the
// moment; the events that free a job (a slot end, a kill for memory) widen that range, a scan narrows it.
#include "kvs_check.cuh"
#include "kvs_ladder.cuh"
#include "kvs_spec_shape.h"

namespace {

constexpr int ST = 128;                 // threads per CTA: four warps, one evaluation each at a time
constexpr int SWARPS = ST / 32;
constexpr int MAXP = KVS_MAX_PHASES;
constexpr int NEVER = 0x7fffffff;
constexpr u32 NO_ROUND = 0xffffffffu;   // completion rounds are kept as 32-bit unsigned: t + o stays below 2^32

struct SpecShared {
  u128 pw_a[MAXP + 1];
  u128 pw_b[MAXP + 1];
  u32 tau[MAXP], k[MAXP], np[MAXP], hist[MAXP];
  i64 pbase[MAXP + 1];
  int n_phases;
};

// floor(r * tau / k) for r, tau, k below 2^31
__device__ __forceinline__ i64 slot_of(int r, u32 tau, u32 k) {
  const u64 x = static_cast<u64>(static_cast<u32>(r)) * tau;
  return (x >> 32) == 0 ? static_cast<i64>(static_cast<u32>(x) / k) : static_cast<i64>(x / k);
}

__device__ __forceinline__ u32 warp_min_u32(u32 v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, d));
  return v;
}

// Number of ranks r < np with floor(r * tau / k) <= x: r * tau < (x + 1) * k, so ceil((x + 1) * k / tau) of them.
__device__ __forceinline__ int started(i64 x, u32 tau, u32 k, int np) {
  if (x < 0) return 0;
  const u64 v = (static_cast<u64>(x + 1) * k + tau - 1) / tau;
  return v < static_cast<u64>(np) ? static_cast<int>(v) : np;
}

// Bytes of one warp's working storage for instances of at most n jobs: five int arrays (position in the phase's
// list, start of the speculative run or -1, stack of speculative runs as job and completion round,
// participant list) and two byte arrays (class, done flag).
__host__ __device__ inline i64 spec_stride(i64 n) { return (22 * n + 255) & ~static_cast<i64>(255); }

__global__ void __launch_bounds__(ST) k_spec(SpecParams p) {
  __shared__ SpecShared shs[SWARPS];
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  SpecShared& sh = shs[warp];
  const i64 wslot = static_cast<i64>(blockIdx.x) * SWARPS + warp;
  if (wslot >= p.n_warps) return;
  const i64 cap = p.max_jobs;
  if (!KVS_OK_AT((wslot + 1) * spec_stride(cap) - 1, p.scratch_bytes, CHK_SP_SCRATCH)) return;
  unsigned char* const mine = p.scratch + wslot * spec_stride(cap);
  int* const pos_of = reinterpret_cast<int*>(mine);    // position of a job in the current phase's list
  int* const sst = pos_of + cap;
  int* const stk_job = sst + cap;
  int* const stk_fin = stk_job + cap;                    // round in which the entry's run would complete
  int* const list = stk_fin + cap;
  unsigned char* const cls = reinterpret_cast<unsigned char*>(list + cap);
  unsigned char* const done = cls + cap;

  for (;;) {
    ull slot = 0;
    if (lane == 0) slot = atomicAdd(p.counter, 1ull);
    slot = __shfl_sync(0xffffffffu, slot, 0);
    if (slot >= (p.left_list ? *p.left_count : static_cast<ull>(p.n_list))) return;
    const i64 e = p.left_list ? p.left_list[slot] : p.eval_list[slot];
    if (p.status[e] != 0) continue;                     // the slicing schedule was not formed or not stored in full
    const kvs_setting st = p.settings[e];
    const i64 lo = p.job_off[st.instance];
    const int n = static_cast<int>(p.job_off[st.instance + 1] - lo);
    const InstStats stats = p.stats[st.instance];
    const i64 M = st.M;
    const i64 s_bar = st.s_bar >= 0 ? st.s_bar : stats.s_max;
    const i64 X = M - s_bar;
    const int32_t* const S = p.s + lo;
    const int32_t* const O = p.o + lo;
    int32_t* const prof = p.profile + p.profile_off[e];
    int32_t* const js = p.job_start + p.job_out_off[e];
    int32_t* const jc = p.job_completion + p.job_out_off[e];
    const int H = static_cast<int>(p.horizon[e]);       // of the slicing schedule; within the profile's capacity (status 0)
    if (!KVS_OK_AT(H, p.profile_off[e + 1] - p.profile_off[e] + 1, CHK_SP_PROF) || !KVS_OK_AT(n, cap + 1, CHK_SP_JOB)) continue;
    if (n == 0) continue;

    // ---- phase table: ladder, classes, participants, first round of every phase ----
    ladder32(sh, X, st.alpha_num, st.alpha_den, st.beta0, static_cast<u32>(s_bar), static_cast<u32>(M));
    const int L = sh.n_phases;
    for (int q = lane; q < L; q += 32) sh.hist[q] = 0;
    __syncwarp();
    const bool pow2 = st.alpha_num == 2 && st.alpha_den == 1 && st.beta0 <= 0;
    for (int i = lane; i < n; i += 32) {
      const u32 oi = static_cast<u32>(O[i]);
      const int c = pow2 ? class_pow2(static_cast<u32>(X), oi) : class_of(sh.tau, L, oi);
      cls[i] = static_cast<unsigned char>(c);
      done[i] = 0; pos_of[i] = i; sst[i] = -1; list[i] = i;
      atomicAdd(&sh.hist[c], 1u);
    }
    __syncwarp();
    if (lane == 0) {
      u32 later = static_cast<u32>(n);
      i64 b = 0;
      for (int q = 0; q < L; ++q) {
        sh.np[q] = later;                               // jobs of class q or later take part in phase q
        sh.pbase[q] = b;
        if (later > 0) b += slot_of(static_cast<int>(later) - 1, sh.tau[q], sh.k[q]) + sh.tau[q];
        later -= sh.hist[q];
      }
      sh.pbase[L] = b;
    }
    __syncwarp();

    // ---- the simulation ----
    int ph = 0, np = n;                                 // phase that holds round t; its participants
    u32 tau_c = sh.tau[0], k_c = sh.k[0];
    i64 base_c = 0;
    int rs = 0, re = 0;                                 // ranks of the next run start and of the next slot end
    i64 ns = 0, ne = tau_c;                             // their rounds
    i64 A = 0;                                          // speculative runs hold A + t * cnt tokens in round t
    int cnt = 0, top = 0;                               // running speculative runs; entries on the stack (some stale)
    u32 next_comp = NO_ROUND;                           // no speculative run completes before this round
    int fpos = 0, fhi = n;
    int cj = -1, cs = 0;                                // the free job at fpos and its prompt length, while known (cj = -2: none is free)
    int left = n;
    i64 flow = 0, steps = 0, runs = 0, peak = 0;
    int hmax = 0;
    int Bw = 0;                                         // lane l holds the plan's memory of round (t & ~31) + l
    for (int t = 0; t <= H; ++t) {
      // (1) speculative completions
      const u32 tu = static_cast<u32>(t);
      if (tu == next_comp) {
        u32 nc = NO_ROUND;
        for (int g0 = 0; g0 < top; g0 += 128) {         // four chunks' completion rounds are loaded together
          u32 fq[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) fq[c] = g0 + 32 * c + lane < top ? static_cast<u32>(stk_fin[g0 + 32 * c + lane]) : NO_ROUND;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int q = g0 + 32 * c + lane;
            const u32 f = fq[c];
            if (f > tu) nc = min(nc, f);                // stale entries included: they cost one empty scan at most
            if (__ballot_sync(0xffffffffu, f == tu) == 0) continue;
            bool fin = false;
            int j = 0, s0 = 0;
            if (f == tu) {
              j = stk_job[q];
              if (!KVS_OK_AT(j, n, CHK_SP_JOB)) j = 0;
              s0 = t - O[j];
              fin = sst[j] == s0;                       // a live entry
            }
            const unsigned fm = __ballot_sync(0xffffffffu, fin);
            if (fm) {
              if (fin) { done[j] = 1; sst[j] = -1; js[j] = s0; jc[j] = t; }
              const i64 dA = warp_sum(fin ? static_cast<i64>(S[j]) + 1 - s0 : static_cast<i64>(0));
              const i64 dS = warp_sum(fin ? static_cast<i64>(O[j]) : static_cast<i64>(0));
              const int kf = __popc(fm);
              A -= dA; steps += dS; flow += static_cast<i64>(kf) * t;
              cnt -= kf; left -= kf; runs += kf;
              hmax = max(hmax, t);
            }
          }
        }
        next_comp = warp_min_u32(nc);
        __syncwarp();
      }
      // slots that have ended: a job killed at the end of its slot is free again.  The ranks whose slots end by
      // round t are [re, started(t - tau)); only those before fpos can lower it.
      if (ne <= t) {
        const int eend = started(static_cast<i64>(t) - tau_c - base_c, tau_c, k_c, np);
        // the ranks [re, eend) are free now unless done or running speculatively; those before fpos are looked at
        // here (the known candidate stays the lowest free job if none of them is), the others lie in the range
        const int lim = min(eend, fpos);
        for (int r0 = re; r0 < lim; r0 += 32) {
          const int r = r0 + lane;
          bool fr = false;
          if (r < lim && KVS_OK_AT(r, n, CHK_SP_LIST)) {
            const int j = list[r];
            if (KVS_OK_AT(j, n, CHK_SP_JOB)) fr = !done[j] && sst[j] < 0;
          }
          const unsigned hit = __ballot_sync(0xffffffffu, fr);
          if (hit) { fpos = r0 + __ffs(static_cast<int>(hit)) - 1; cj = -1; break; }
        }
        if (eend > fhi && (cj == -1 || eend > lim)) fhi = eend;
        re = eend;
        ne = re < np ? base_c + slot_of(re, tau_c, k_c) + tau_c : static_cast<i64>(NEVER) * 2;
      }
      // the next phase begins: its participants are the jobs of a later class, in index order
      if (rs >= np && ph + 1 < L && sh.np[ph + 1] > 0 && t == sh.pbase[ph + 1]) {
        ++ph;
        int w = 0;
        for (int q0 = 0; q0 < np; q0 += 32) {
          const int q = q0 + lane;
          bool keep = false;
          int j = 0;
          if (q < np && KVS_OK_AT(q, n, CHK_SP_LIST)) { j = list[q]; keep = KVS_OK_AT(j, n, CHK_SP_JOB) && cls[j] >= ph; }
          const unsigned m = __ballot_sync(0xffffffffu, keep);
          __syncwarp();
          if (keep) { const int d = w + __popc(m & lt_mask); list[d] = j; pos_of[j] = d; }
          w += __popc(m);
          __syncwarp();
        }
        np = w;
        tau_c = sh.tau[ph]; k_c = sh.k[ph]; base_c = sh.pbase[ph];
        rs = 0; re = 0; ns = base_c; ne = base_c + tau_c;
        fpos = 0; fhi = np; cj = -1;
      }
      // (2) pipeline runs that start now: ranks [rs, started(t)), 32 at a time (they concern different jobs)
      if (ns <= t) {
        const int rend = started(static_cast<i64>(t) - base_c, tau_c, k_c, np);
        bool cand_started = false;                      // a job that starts may be the known candidate
        for (int r0 = rs; r0 < rend; r0 += 32) {
          const int r = r0 + lane;
          bool act = r < rend && KVS_OK_AT(r, n, CHK_SP_LIST);
          int j = 0, oj = 0, sj = 0, s0 = -1;
          bool dn = false;
          if (act) { j = list[r]; act = KVS_OK_AT(j, n, CHK_SP_JOB); }
          if (act) { oj = O[j]; sj = S[j]; dn = done[j] != 0; s0 = sst[j]; }
          if (cj >= 0 && __ballot_sync(0xffffffffu, act && j == cj)) cand_started = true;
          const int len = oj < static_cast<int>(tau_c) ? oj : static_cast<int>(tau_c);
          const bool run = act && !dn, drop = act && dn;
          const bool kill = run && s0 >= 0;             // its speculative run is killed; the stack entry goes stale
          const bool comp = run && len == oj;
          const unsigned km = __ballot_sync(0xffffffffu, kill);
          if (km) {
            A -= warp_sum(kill ? static_cast<i64>(sj) + 1 - s0 : static_cast<i64>(0));
            steps += warp_sum(kill ? static_cast<i64>(t - s0) : static_cast<i64>(0));
            cnt -= __popc(km);
            runs += __popc(__ballot_sync(0xffffffffu, kill && t > s0));
          }
          const unsigned rm = __ballot_sync(0xffffffffu, run);
          if (rm) {
            steps += warp_sum(run ? static_cast<i64>(len) : static_cast<i64>(0));
            runs += __popc(rm);
            if (run) {
              sst[j] = -1;
              if (comp) { done[j] = 1; js[j] = t; jc[j] = t + len; }
            }
            const unsigned cm = __ballot_sync(0xffffffffu, comp);
            if (cm) {
              left -= __popc(cm);
              flow += warp_sum(comp ? static_cast<i64>(t + len) : static_cast<i64>(0));
              hmax = max(hmax, warp_max(comp ? t + len : 0));
            }
          }
          // dropped from the plan: short ramps lane by lane, long ones by the whole warp; the rounds of the
          // window held in registers are corrected there (the round of lane l is t - (t & 31) + l)
          unsigned dm = __ballot_sync(0xffffffffu, drop);
          if (dm) {
            if (drop && len <= 64)
              for (int u = 0; u < len; ++u)
                if (KVS_OK_AT(t + u, H, CHK_SP_DROP)) atomicSub(&prof[t + u], sj + u + 1);
            unsigned lm = __ballot_sync(0xffffffffu, drop && len > 64);
            while (lm) {
              const int src = __ffs(static_cast<int>(lm)) - 1;
              lm &= lm - 1u;
              const int ls = __shfl_sync(0xffffffffu, len, src), ss = __shfl_sync(0xffffffffu, sj, src);
              for (int u = lane; u < ls; u += 32)
                if (KVS_OK_AT(t + u, H, CHK_SP_DROP)) atomicSub(&prof[t + u], ss + u + 1);
            }
            if ((t & 31) != 0) {                        // at a window's first round the window is loaded afterwards
              const int u = lane - (t & 31);            // this lane's round, counted from t
              while (dm) {
                const int src = __ffs(static_cast<int>(dm)) - 1;
                dm &= dm - 1u;
                const int ls = __shfl_sync(0xffffffffu, len, src), ss = __shfl_sync(0xffffffffu, sj, src);
                if (u >= 0 && u < ls) Bw -= ss + u + 1;
              }
            }
          }
        }
        __syncwarp();
        if (cand_started) cj = -1;
        rs = rend;
        ns = rs < np ? base_c + slot_of(rs, tau_c, k_c) : static_cast<i64>(NEVER) * 2;
      }
      if (t == H) break;                                // nothing runs in round H; only completions were due
      if (left == 0) {
        // Every job is done, so every run the pipeline has yet to start is dropped: what is left of the plan are
        // the runs in progress, which are completing runs of ranks between the two cursors (a killed run in
        // progress would belong to an unfinished job).  Such a run's completion round lies beyond t and it began o earlier.
        __syncwarp();
        for (int u = t + lane; u < H; u += 32) prof[u] = 0;
        __syncwarp();
        for (int r = re; r < rs; ++r) {
          const int j = list[r];
          if (!KVS_OK_AT(j, n, CHK_SP_JOB)) continue;
          const int end = jc[j];                        // beyond t only for a completing run of the pipeline in progress
          if (end > t && KVS_OK_AT(end, H + 1, CHK_SP_PROF)) {
            const int first = end - O[j], sj = S[j];
            for (int u = t + lane; u < end; u += 32) prof[u] += sj + (u - first) + 1;
            __syncwarp();
          }
        }
        i64 pk = 0;
        for (int u = t + lane; u < hmax; u += 32) pk = max_i64(pk, __ldcg(prof + u));
        peak = max_i64(peak, warp_max(pk));
        break;
      }
      if ((t & 31) == 0) {                              // the plan's next 32 rounds, past the first-level cache: other lanes' atomics wrote them
        __syncwarp();
        const int u = t + lane;
        Bw = u < H ? __ldcg(prof + u) : 0;
      }
      const i64 B = __shfl_sync(0xffffffffu, Bw, t & 31);
      // (3) the pipeline comes first
      while (cnt > 0 && B + A + static_cast<i64>(t) * cnt > M) {
        int j = -1, s0 = 0;
        while (top > 0) {                               // the live entry nearest to the top
          --top;
          const int jj = stk_job[top];
          if (!KVS_OK_AT(jj, n, CHK_SP_JOB)) continue;
          s0 = static_cast<int>(static_cast<u32>(stk_fin[top]) - static_cast<u32>(O[jj]));
          if (sst[jj] == s0) { j = jj; break; }
        }
        if (j < 0) break;
        __syncwarp();
        A -= static_cast<i64>(S[j]) + 1 - s0;
        --cnt;
        steps += t - s0;
        runs += t > s0 ? 1 : 0;
        if (lane == 0) sst[j] = -1;
        __syncwarp();
        const int a = pos_of[j];                        // free again: it may come before the known candidate
        if (!KVS_OK_AT(a, np, CHK_SP_LIST)) break;
        if (a < fpos) { fpos = a; cj = -1; }
        if (a >= fhi) { fhi = a + 1; if (cj == -2) cj = -1; }
      }
      // (4) first come first served: the free jobs of a window of 32 list entries are admitted together as far as
      // their first rounds fit, in order; the first that does not fit ends the round's admissions
      for (;;) {
        const i64 room = M - (B + A + static_cast<i64>(t) * cnt);
        if (cj == -2 || (cj >= 0 && cs + 1 > room) || room <= 0) break;
        // the jobs in a pipeline run are the ranks whose slot has begun and not ended: [re, rs)
        if (fpos >= re && fpos < rs) fpos = rs;
        if (fpos >= fhi) { fpos = np; fhi = 0; cj = -2; break; }
        const int q = fpos + lane;
        bool fr = false;
        int j = 0, sj = 0;
        if (q < fhi && !(q >= re && q < rs) && KVS_OK_AT(q, n, CHK_SP_LIST)) {
          j = list[q];
          if (KVS_OK_AT(j, n, CHK_SP_JOB)) fr = !done[j] && sst[j] < 0; else j = 0;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, fr);
        if (!hit) { fpos += 32; cj = -1; continue; }
        if (fr) sj = S[j];
        i64 need = fr ? static_cast<i64>(sj) + 1 : 0;   // inclusive prefix sums over the window, in list order
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const i64 y = __shfl_up_sync(0xffffffffu, need, d);
          if (lane >= d) need += y;
        }
        const bool ok = fr && need <= room;
        const unsigned okm = __ballot_sync(0xffffffffu, ok);
        const int m = __popc(okm);
        if (m) {
          if (top + 32 > static_cast<int>(cap) || top > 2 * cnt + 64) {   // mostly stale entries: keep the live ones, in order
            int w = 0;
            for (int q0 = 0; q0 < top; q0 += 32) {
              const int qq = q0 + lane;
              bool live = false;
              int jj = 0, ff = 0;
              if (qq < top) { jj = stk_job[qq]; ff = stk_fin[qq]; live = KVS_OK_AT(jj, n, CHK_SP_JOB) && sst[jj] == static_cast<int>(static_cast<u32>(ff) - static_cast<u32>(O[jj])); }
              const unsigned lm = __ballot_sync(0xffffffffu, live);
              __syncwarp();
              if (live) { const int d = w + __popc(lm & lt_mask); stk_job[d] = jj; stk_fin[d] = ff; }
              w += __popc(lm);
              __syncwarp();
            }
            top = w;
          }
          const u32 fin = ok ? tu + static_cast<u32>(O[j]) : NO_ROUND;
          if (ok) {
            const int d = top + __popc(okm & lt_mask);
            if (KVS_OK_AT(d, cap, CHK_SP_STACK)) { sst[j] = t; stk_job[d] = j; stk_fin[d] = static_cast<int>(fin); }
          }
          __syncwarp();
          top += m;
          A += warp_sum(ok ? static_cast<i64>(sj) + 1 - t : static_cast<i64>(0));
          cnt += m;
          next_comp = min(next_comp, warp_min_u32(fin));
        }
        const unsigned failed = hit & ~okm;
        if (failed) {                                   // the first free job that does not fit is the candidate from now on
          const int src = __ffs(static_cast<int>(failed)) - 1;
          fpos += src;
          cj = __shfl_sync(0xffffffffu, j, src);
          cs = __shfl_sync(0xffffffffu, sj, src);
          break;
        }
        fpos += 32; cj = -1;
      }
      // (5) the round's memory
      const i64 mem = B + A + static_cast<i64>(t) * cnt;
      if (lane == 0 && KVS_OK_AT(t, H, CHK_SP_PROF)) prof[t] = static_cast<int32_t>(mem);
      peak = max_i64(peak, mem);
      if (cnt == 0) top = 0;                            // only stale entries are left
    }
    __syncwarp();
    if (lane == 0) {
      if (p.peak) p.peak[e] = peak;
      if (p.flow) p.flow[e] = flow;
      if (p.job_steps) p.job_steps[e] = steps;
      if (p.n_runs) p.n_runs[e] = runs;
      if (p.n_unfinished) p.n_unfinished[e] = left;
      p.horizon[e] = hmax;
      if (p.feasible) p.feasible[e] = peak <= M ? 1 : 0;
    }
    __syncwarp();
  }
}

// ---- the same simulation with its state in shared memory --------------------------------------------
//
// What bounds a simulation is the chain of steps of its one warp, so what counts is the number of rounds at which the warp has to
// stop, the dependent instructions of each stop, and the evaluations that an SM has in flight.  Instances of at most some 25,000
// jobs (lengths below 2^16) fit on chip: 4 bytes a job of prompt and response lengths, which the warps of a CTA share (up to four
// evaluations of one instance, see kvs_spec_shape), and per evaluation 4 bytes a job - start of the speculative run, stack entry - and two bits.  Besides:
//   - a job that is free to start a speculative run has its bit set in a map by job index: the order of the participants is that
//     of the indices and whoever is no participant any more is done, so the lowest free job is the first bit, found by one
//     16-byte load a lane over 4,096 jobs; slot ends and kills set a bit and know at once whether it is the lowest;
//   - the rounds are taken 32 at a time.  Where a window's pipeline runs are few, all of them are looked at when it begins: those
//     of jobs that have completed are dropped there and then, together, and neither their starts nor their slot ends stop the warp;
//   - a run dropped from the plan is not subtracted from the profile round by round: those in progress hold Ad + t * Cd tokens, with
//     starts and ends in a ring of 256 to 1,024 rounds, ends beyond it in a list of FAR_SETS entries a lane (beyond that in memory);
//   - the participants' list lies in memory: it is read in order, the next 32 entries ahead of time;
//   - the rounds up to the next event are written together: nothing can happen in a round in which nothing starts or ends, the
//     memory stays within M and the first free job does not fit;
//   - the stack keeps the earliest completion of every 64 entries, so that a completion looks at few entries;
//   - sums that nothing in the simulation depends on are kept per lane.
// Starts are kept modulo 65,535: a speculative run lasts less than that.
// 512 evaluations (64 instances of 5,000 to 10,000 jobs, eight budgets), four per CTA and all in flight: 17.6 ms, the chain of the longest
// one.  With every run's start and slot end a stop, list scans of 32 positions for the lowest free job and two evaluations per SM: 56.7 ms.

constexpr int FAR_SETS = 6;
constexpr u32 IDLE = 0xffffu;            // sst: not running speculatively
constexpr u32 MODT = 65535u;
constexpr int LOOK_AHEAD = 1024;         // runs that may start in a window whose runs are looked at together: a mask of 32 per lane

// The phase table of one warp; the powers of the ladder lie where the stack will be.
struct alignas(16) SpecTable {
  u32 tau[MAXP], k[MAXP], np[MAXP], hist[MAXP];
  int pbase[MAXP + 1];
  int n_phases;
  u128 *pw_a, *pw_b;
};

static_assert(sizeof(SpecTable) == SPEC_TABLE_BYTES && 2 * (MAXP + 1) * sizeof(u128) == SPEC_POWERS_BYTES, "bytes of a warp's state");

// floor(x / d) by the multiplication with floor(2^64 / d) + 1 where x is below 2^32 (see slot_mul in kvs_fused.cu)
__device__ __forceinline__ u32 div_by(u64 x, u32 d, u64 dinv) {
  if ((x >> 32) == 0) return d == 1 ? static_cast<u32>(x) : static_cast<u32>(__umul64hi(x, dinv));
  return static_cast<u32>(x / d);
}
__device__ __forceinline__ u64 inverse_of(u32 d) { return d >= 2 ? ~0ull / d + 1ull : 0ull; }

// What one warp keeps of the phase that holds the current round.
struct SpecPhase {
  u32 tau, k;
  u64 tau_inv, k_inv;
  int np;
  int base;
  bool ahead;               // fewer than LOOK_AHEAD runs start in a window
  __device__ __forceinline__ int start_of(int r) const { return base + static_cast<int>(div_by(static_cast<u64>(static_cast<u32>(r)) * tau, k, k_inv)); }
  // ranks that start x rounds after the phase's first round or earlier
  __device__ __forceinline__ int started(int x) const {
    if (x < 0) return 0;
    const u64 v = static_cast<u64>(static_cast<u32>(x) + 1u) * k + (tau - 1u);
    if ((v >> 32) == 0) return min(static_cast<int>(min(div_by(v, tau, tau_inv), 0x7fffffffu)), np);
    const u64 q = v / tau;
    return q < static_cast<u64>(np) ? static_cast<int>(q) : np;
  }
};

__global__ void __launch_bounds__(32 * SPEC_WARPS) k_spec_smem(SpecParams p, int n_cap, int ring_rounds) {
  extern __shared__ __align__(16) unsigned char raw[];
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int m = smem_jobs(n_cap);
  u32* const lengths = reinterpret_cast<u32*>(raw);     // response length << 16 | prompt length
  unsigned char* at = raw + smem_lengths_bytes(n_cap) + warp * smem_state_bytes(n_cap, ring_rounds);
  SpecTable& sh = *reinterpret_cast<SpecTable*>(at); at += sizeof(SpecTable);
  u32* const ring_a = reinterpret_cast<u32*>(at); at += ring_rounds * 4;
  u32* const ring_c = reinterpret_cast<u32*>(at); at += ring_rounds * 4;
  const int ring_mask = ring_rounds - 1;
  unsigned char* const stk_at = at; at += smem_stack_bytes(m);
  unsigned short* const stk = reinterpret_cast<unsigned short*>(stk_at);  // jobs in order of their starts; an entry whose job is not running is stale, and so is one with another above it
  u32* const free_map = reinterpret_cast<u32*>(at); at += m / 8;          // neither done nor running
  u32* const done = reinterpret_cast<u32*>(at); at += m / 8;
  unsigned short* const sst = reinterpret_cast<unsigned short*>(at); at += m * 2;
  u32* const first_fin = reinterpret_cast<u32*>(at);                     // no run of the block's entries completes before this round
  const i64* const group = p.groups + SPEC_WARPS * static_cast<i64>(blockIdx.x);
  const i64 mine = group[warp];                         // -1: no evaluation for this warp
  const i64 inst = p.settings[group[0]].instance;
  const i64 lo = p.job_off[inst];
  const InstStats stats = p.stats[inst];
  // the memory of a round, pipeline and speculative runs before any is killed, stays below 2^32
  // (the warps decide together: all of them load the lengths)
  i64 M_most = 0;
  for (int v = 0; v < static_cast<int>(blockDim.x >> 5); ++v)
    if (group[v] >= 0) M_most = max_i64(M_most, p.settings[group[v]].M);
  const int n = stats.flags ? 0 : static_cast<int>(p.job_off[inst + 1] - lo);
  if (n > n_cap || stats.o_max >= static_cast<int>(MODT) || stats.s_max >= 65536 || M_most >= (1ll << 30)) {
    if (lane == 0 && mine >= 0) p.left_list[atomicAdd(p.left_count, 1ull)] = mine;
    return;
  }
  const u32 among_all = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;     // (the stride as a parameter or a variable of its own: 17.74 instead of 17.64 ms)
  unsigned short* const list = reinterpret_cast<unsigned short*>(p.scratch) + static_cast<i64>(among_all) * m;   // spec_list_bytes a CTA
  if (!KVS_OK_AT((static_cast<i64>(among_all) + 1) * m * 2 - 1, p.scratch_bytes, CHK_SP_SCRATCH)) return;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    lengths[i] = static_cast<u32>(p.o[lo + i]) << 16 | static_cast<u32>(p.s[lo + i]);
  }
  __syncthreads();
  if (mine < 0 || n == 0) return;
  const i64 e = mine;
  if (p.status[e] != 0) return;                         // the slicing schedule was not formed or not stored in full
  const kvs_setting set = p.settings[e];
  const i64 M = set.M;
  const i64 s_bar = set.s_bar >= 0 ? set.s_bar : stats.s_max;
  const i64 X = M - s_bar;
  int32_t* const prof = p.profile + p.profile_off[e];
  int32_t* const js = p.job_start + p.job_out_off[e];
  int32_t* const jc = p.job_completion + p.job_out_off[e];
  const int H = static_cast<int>(p.horizon[e]);         // of the slicing schedule; within the profile's capacity (status 0)
  if (!KVS_OK_AT(H, p.profile_off[e + 1] - p.profile_off[e] + 1, CHK_SP_PROF)) return;

  // ---- phase table: ladder, classes, participants, first round of every phase ----
  if (lane == 0) { sh.pw_a = reinterpret_cast<u128*>(stk_at); sh.pw_b = sh.pw_a + MAXP + 1; }
  __syncwarp();
  ladder32(sh, X, set.alpha_num, set.alpha_den, set.beta0, static_cast<u32>(s_bar), static_cast<u32>(M));
  const int L = sh.n_phases;
  for (int q = lane; q < L; q += 32) sh.hist[q] = 0;
  for (int i = lane; i < ring_rounds; i += 32) { ring_a[i] = 0; ring_c[i] = 0; }
  for (int i = lane; i < m / 32; i += 32) {
    const int room = n - 32 * i;
    done[i] = 0;
    if (i < m / STK_BLK) first_fin[i] = NO_ROUND;
    free_map[i] = room >= 32 ? 0xffffffffu : (room > 0 ? (1u << room) - 1u : 0u);
  }
  __syncwarp();
  const bool pow2 = set.alpha_num == 2 && set.alpha_den == 1 && set.beta0 <= 0;
  for (int i = lane; i < n; i += 32) {
    const u32 oi = lengths[i] >> 16;
    atomicAdd(&sh.hist[pow2 ? class_pow2(static_cast<u32>(X), oi) : class_of(sh.tau, L, oi)], 1u);
    sst[i] = static_cast<unsigned short>(IDLE);
  }
  __syncwarp();
  if (lane == 0) {
    u32 later = static_cast<u32>(n);
    i64 b = 0;
    for (int q = 0; q < L; ++q) {
      sh.np[q] = later;                                 // jobs of class q or later take part in phase q
      sh.pbase[q] = static_cast<int>(b);
      if (later > 0) b += slot_of(static_cast<int>(later) - 1, sh.tau[q], sh.k[q]) + sh.tau[q];
      later -= sh.hist[q];
    }
    sh.pbase[L] = static_cast<int>(b);
  }
  __syncwarp();
  const u32 Mu = static_cast<u32>(M);
  auto is_done = [&](u32 j) { return (done[j >> 5] >> (j & 31u) & 1u) != 0; };

  // ---- the simulation ----
  SpecPhase ph;
  int phase = 0;
  auto enter = [&](int q, int participants) {
    ph.tau = sh.tau[q]; ph.k = sh.k[q];
    ph.tau_inv = inverse_of(ph.tau); ph.k_inv = inverse_of(ph.k);
    ph.np = participants;
    ph.base = sh.pbase[q];
    // 32 rounds hold at most ceil(32 k / tau) + 1 starts, and as many slot ends
    ph.ahead = static_cast<u64>(ph.k) * 32u <= static_cast<u64>(ph.tau) * (LOOK_AHEAD - 2);
  };
  enter(0, n);
  int rs = 0, re = 0;                                   // ranks behind the runs (and the slot ends) that have been looked at
  int ns = 0, ne = static_cast<int>(ph.tau);            // rounds of the next run start and of the next slot end
  // The runs of 32 consecutive ranks that start next, one a lane: job, response, prompt + 1, first round, and which of them the warp
  // still has to stop for; the same for the slot ends.  Where the window has been looked at, lane c holds the mask of its c-th 32.
  u32 start_job = 0, start_o = 0, start_s1 = 0, end_job = 0;
  int start_at = 0, end_at = 0, start_first = 0, end_first = 0;
  unsigned start_mask = 0, end_mask = 0, start_masks = 0, end_masks = 0;
  bool all_take_part = true;                            // rank = job index: no list yet
  u32 ahead_start = 0, ahead_end = 0;                   // list entries of ranks rs + lane and re + lane, read ahead
  // a job number that was read from the list or the stack (checked build: 0 if it is none)
  auto job_at = [&](u32 j) { return KVS_OK_AT(j, n, CHK_SP_JOB) ? j : 0u; };
  auto list_at = [&](int r) { return KVS_OK_AT(r, n, CHK_SP_LIST) ? job_at(list[r]) : 0u; };
  // job of rank r < np
  auto job_of = [&](int r) { return all_take_part ? job_at(static_cast<u32>(r)) : list_at(r); };
  int phase_at = L > 1 && sh.np[1] > 0 ? sh.pbase[1] : NEVER;   // first round of the next phase
  u32 A = 0;                                            // speculative runs hold A + t * cnt tokens in round t (modulo 2^32)
  int cnt = 0, top = 0;                                 // running speculative runs; entries on the stack (some stale)
  u32 Ad = 0, Cd = 0;                                   // dropped runs in progress at the end of the current window
  u32 far_v[FAR_SETS], far_c[FAR_SETS];                 // those of them that end beyond the ring (end 0: none)
  int far_end[FAR_SETS];
#pragma unroll
  for (int f = 0; f < FAR_SETS; ++f) far_v[f] = far_c[f] = static_cast<u32>(far_end[f] = 0);
  int far_next = NEVER;                                 // the earliest of them
  u32 next_comp = NO_ROUND;                             // no speculative run completes before this round
  int fj = 0;                                           // no job below is free
  int cj = -1, cs = 0;                                  // the lowest free job and its prompt length, while known (then fj = cj; -2: none is free)
  int left = n;
  i64 flow = 0, steps = 0;                              // flow, steps, runs, hmax, peak: per lane
  u32 runs = 0, peak = 0;
  int hmax = 0;
  int Bw = 0;                                           // lane l holds the plan's memory of round (t & ~31) + l,
  int Bn = lane < H ? __ldcg(prof + lane) : 0;          // that of the window after it (past the first-level cache: atomics wrote it)
  u32 tm = 0;                                           // t modulo MODT

  // The next 32 of the window's runs with one that the warp stops for.
  auto next_starts = [&]() {
    const unsigned chunks = __ballot_sync(0xffffffffu, start_masks != 0);
    if (!chunks) { ns = NEVER; return; }
    const int c = __ffs(static_cast<int>(chunks)) - 1, r = start_first + 32 * c + lane;
    start_mask = __shfl_sync(0xffffffffu, start_masks, c);
    start_job = job_of(min(r, rs - 1));
    const u32 so = lengths[start_job];
    start_o = so >> 16; start_s1 = (so & 0xffffu) + 1u;
    start_at = ph.start_of(r);
    if (lane == c) start_masks = 0;
    ns = __shfl_sync(0xffffffffu, start_at, __ffs(static_cast<int>(start_mask)) - 1);
  };
  auto next_ends = [&]() {
    const unsigned chunks = __ballot_sync(0xffffffffu, end_masks != 0);
    if (!chunks) { ne = NEVER; return; }
    const int c = __ffs(static_cast<int>(chunks)) - 1, r = end_first + 32 * c + lane;
    end_mask = __shfl_sync(0xffffffffu, end_masks, c);
    end_job = job_of(min(r, re - 1));
    end_at = ph.start_of(r) + static_cast<int>(ph.tau);
    if (lane == c) end_masks = 0;
    ne = __shfl_sync(0xffffffffu, end_at, __ffs(static_cast<int>(end_mask)) - 1);
  };
  // c dropped runs that last beyond the ring, with v = sum of s + 1 - start, that are in progress at the end of window w: into the
  // list, false if it is full.
  auto keep_far = [&](u32 v, u32 c, int end) {
#pragma unroll
    for (int f = 0; f < FAR_SETS; ++f) {
      const unsigned room = __ballot_sync(0xffffffffu, far_end[f] == 0);
      if (room) {
        if (lane == __ffs(static_cast<int>(room)) - 1) { far_v[f] = v; far_c[f] = c; far_end[f] = end; }
        far_next = min(far_next, end);
        return true;
      }
    }
    return false;
  };
  // Then they are taken out of the window after w, which is in registers, and of the rounds behind it.
  auto drop_in_memory = [&](int w, u32 v, u32 c, int end) {
    const int u = w + 32 + lane;
    if (u < end) Bn -= static_cast<int>(v + c * static_cast<u32>(u));
    for (int x = u + 32; x < end; x += 32)              // always the rounds of one lane: its later read follows
      if (KVS_OK_AT(x, H, CHK_SP_DROP)) atomicSub(&prof[x], static_cast<int>(v + c * static_cast<u32>(x)));
  };
  // Runs dropped in round t of window w.
  auto drop_now = [&](int w, int t, u32 v, u32 c, int end) {
    const int u = w + lane;
    if (u >= t && u < end) Bw -= static_cast<int>(v + c * static_cast<u32>(u));
    if (end <= w + 32) return;
    if (end < w + ring_rounds) {
      Ad += v; Cd += c;
      if (lane == 0) { ring_a[end & ring_mask] += v; ring_c[end & ring_mask] += c; }
      __syncwarp();
    } else if (keep_far(v, c, end)) {
      Ad += v; Cd += c;
    } else {
      drop_in_memory(w, v, c, end);
    }
  };
  // Looks at the runs that start and the slots that end from round t to the end of its window w: drops the runs of jobs that are
  // done.  read: the first 32 list entries of each have been read ahead.
  auto look_ahead = [&](int w, int t, bool read) {
    const int r_hi = ph.started(w + 31 - ph.base);
    start_first = rs; start_masks = 0; start_mask = 0; ns = NEVER;
    for (int c = 0, r0 = rs; r0 < r_hi; ++c, r0 += 32) {
      const int r = r0 + lane;
      const bool on = r < r_hi;
      const u32 j = !on ? 0u : (all_take_part ? job_at(static_cast<u32>(r)) : (read && c == 0 ? ahead_start : list_at(r)));
      const u32 so = lengths[j], o = so >> 16, s1 = (so & 0xffffu) + 1u;
      const bool drop = on && is_done(j);
      const int q = ph.start_of(r);
      const unsigned live = __ballot_sync(0xffffffffu, on && !drop);
      if (live && ns == NEVER) {
        start_mask = live;
        start_job = j; start_o = o; start_s1 = s1; start_at = q;
        ns = __shfl_sync(0xffffffffu, q, __ffs(static_cast<int>(live)) - 1);
      } else if (lane == c) {
        start_masks = live;
      }
      if (live == 0xffffffffu) continue;
      const int end = q + static_cast<int>(min(o, ph.tau));
      const u32 v = s1 - static_cast<u32>(q);
      const bool far = end >= w + ring_rounds;
      if (drop && !far) {
        atomicSub(&ring_a[q & ring_mask], v); atomicSub(&ring_c[q & ring_mask], 1u);
        atomicAdd(&ring_a[end & ring_mask], v); atomicAdd(&ring_c[end & ring_mask], 1u);
      }
      unsigned fm = __ballot_sync(0xffffffffu, drop && far);
      while (fm) {
        const int src = __ffs(static_cast<int>(fm)) - 1;
        fm &= fm - 1u;
        const u32 vs = __shfl_sync(0xffffffffu, v, src);
        const int qs = __shfl_sync(0xffffffffu, q, src), es = __shfl_sync(0xffffffffu, end, src);
        if (keep_far(vs, 1u, es)) {
          if (lane == 0) { ring_a[qs & ring_mask] -= vs; ring_c[qs & ring_mask] -= 1u; }
        } else {
          if (w + lane >= qs) Bw -= static_cast<int>(vs + static_cast<u32>(w + lane));
          drop_in_memory(w, vs, 1u, es);
        }
        __syncwarp();
      }
    }
    rs = r_hi;
    const int e_hi = ph.started(w + 31 - static_cast<int>(ph.tau) - ph.base);
    end_first = re; end_masks = 0; end_mask = 0; ne = NEVER;
    for (int c = 0, r0 = re; r0 < e_hi; ++c, r0 += 32) {
      const int r = r0 + lane;
      const bool on = r < e_hi;
      const u32 j = !on ? 0u : (all_take_part ? job_at(static_cast<u32>(r)) : (read && c == 0 ? ahead_end : list_at(r)));
      const unsigned live = __ballot_sync(0xffffffffu, on && !is_done(j));
      if (live && ne == NEVER) {
        end_mask = live;
        end_job = j;
        end_at = ph.start_of(r) + static_cast<int>(ph.tau);
        ne = __shfl_sync(0xffffffffu, end_at, __ffs(static_cast<int>(live)) - 1);
      } else if (lane == c) {
        end_masks = live;
      }
    }
    re = e_hi;
    if (!all_take_part) {
      if (rs + lane < ph.np) ahead_start = list_at(rs + lane);
      if (re + lane < ph.np) ahead_end = list_at(re + lane);
    }
    __syncwarp();
  };
  // Takes the starts and ends of dropped runs in window w out of the ring; a, c: dropped runs in progress at its beginning.
  auto apply_ring = [&](int w, u32 a, u32 c) {
    const int u = w + lane, x = u & ring_mask;
    u32 ea = ring_a[x], ec = ring_c[x];
    if (__any_sync(0xffffffffu, (ea | ec) != 0)) {
      ring_a[x] = 0;
      ring_c[x] = 0;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const u32 ya = __shfl_up_sync(0xffffffffu, ea, d), yc = __shfl_up_sync(0xffffffffu, ec, d);
        if (lane >= d) { ea += ya; ec += yc; }
      }
      Ad -= __shfl_sync(0xffffffffu, ea, 31);
      Cd -= __shfl_sync(0xffffffffu, ec, 31);
    }
    Bw -= static_cast<int>((a - ea) + static_cast<u32>(u) * (c - ec));
    __syncwarp();
  };
  auto running_for = [&](u32 start_m) { return tm >= start_m ? tm - start_m : tm + MODT - start_m; };   // rounds since a start
  auto prompt = [&](int j) { return static_cast<int>(lengths[j] & 0xffffu); };
  // Job j, of prompt length s0, has become free.
  auto freed = [&](int j, u32 s0) { if (cj == -2 || j < fj) { fj = j; cj = j; cs = static_cast<int>(s0); } };
  // The lowest free job, -1 if there is none.
  auto first_free = [&]() {
    for (int b = (fj >> 5) & ~3; b < m / 32; b += 128) {
      const int w = b + 4 * lane;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (w < m / 32) v = *reinterpret_cast<const uint4*>(free_map + w);
      const u32 bits = v.x ? v.x : (v.y ? v.y : (v.z ? v.z : v.w));
      const int word = w + (v.x ? 0 : (v.y ? 1 : (v.z ? 2 : 3)));
      const unsigned hit = __ballot_sync(0xffffffffu, bits != 0);
      if (hit) return __shfl_sync(0xffffffffu, 32 * word + __ffs(static_cast<int>(bits)) - 1, __ffs(static_cast<int>(hit)) - 1);
    }
    return -1;
  };
  // Keeps the live entries of the stack, in order (of every running job the uppermost one, whose place waits in job_start), and forms the
  // earliest completion of every block of entries again.
  auto purge = [&](int t) {
    for (int b = lane; b * STK_BLK < top; b += 32) first_fin[b] = NO_ROUND;
    __syncwarp();
    int w = 0;
    constexpr int U = 4;
    for (int q0 = 0; q0 < top; q0 += 32 * U) {
      u32 j[U], sm[U];
      int place[U];
#pragma unroll
      for (int i = 0; i < U; ++i) {
        const int q = q0 + 32 * i + lane;
        j[i] = q < top && KVS_OK_AT(q, m, CHK_SP_STACK) ? job_at(stk[q]) : 0u;
        sm[i] = q < top ? sst[j[i]] : IDLE;
        place[i] = js[j[i]];
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < U; ++i) {
        const bool live = sm[i] != IDLE && place[i] == q0 + 32 * i + lane;
        const unsigned lm = __ballot_sync(0xffffffffu, live);
        const int d = w + __popc(lm & lt_mask);
        if (live && KVS_OK_AT(d, m, CHK_SP_STACK)) {
          stk[d] = static_cast<unsigned short>(j[i]);
          js[j[i]] = d;
          atomicMin(&first_fin[d / STK_BLK], static_cast<u32>(t) + (lengths[j[i]] >> 16) - running_for(sm[i]));
        }
        w += __popc(lm);
      }
      __syncwarp();
    }
    top = w;
  };
  int t = 0;
  while (t <= H) {
    const u32 tu = static_cast<u32>(t);
    const int w = t & ~31;
    if (t == w && t < H) {
      Bw = Bn;
      Bn = t + 32 + lane < H ? __ldcg(prof + t + 32 + lane) : 0;
      const u32 a = Ad, c = Cd;
      if (far_next < w + ring_rounds) {                 // ends that the ring has come to
        int next = NEVER;
#pragma unroll
        for (int f = 0; f < FAR_SETS; ++f) {
          if (far_end[f] != 0 && far_end[f] < w + ring_rounds) {
            atomicAdd(&ring_a[far_end[f] & ring_mask], far_v[f]); atomicAdd(&ring_c[far_end[f] & ring_mask], far_c[f]);
            far_end[f] = 0;
          }
          if (far_end[f] != 0) next = min(next, far_end[f]);
        }
        far_next = static_cast<int>(__reduce_min_sync(0xffffffffu, static_cast<u32>(next)));
        __syncwarp();
      }
      if (ph.ahead) look_ahead(w, t, true);
      apply_ring(w, a, c);
    }
    // (1) speculative completions
    if (tu == next_comp) {
      u32 nc = NO_ROUND;
      const int blocks = (top + STK_BLK - 1) / STK_BLK;
      for (int b0 = 0; b0 < blocks; b0 += 32) {
        const u32 f = b0 + lane < blocks ? first_fin[b0 + lane] : NO_ROUND;
        if (f > tu) nc = min(nc, f);
        unsigned due = __ballot_sync(0xffffffffu, f <= tu);
        while (due) {
          const int b = b0 + __ffs(static_cast<int>(due)) - 1, q = b * STK_BLK + 2 * lane;
          due &= due - 1u;
          const u32 both = q < top ? *reinterpret_cast<const u32*>(stk + q) : 0u;
          const u32 j0 = job_at(both & 0xffffu), j1 = q + 1 < top ? job_at(both >> 16) : 0u;
          const u32 sm0 = q < top ? sst[j0] : IDLE, sm1 = q + 1 < top ? sst[j1] : IDLE, so0 = lengths[j0], so1 = lengths[j1];
          const u32 ran0 = running_for(sm0), ran1 = running_for(sm1), o0 = so0 >> 16, o1 = so1 >> 16;
          const bool fin0 = sm0 != IDLE && ran0 == o0, fin1 = sm1 != IDLE && ran1 == o1;
          const u32 rest0 = sm0 == IDLE || fin0 ? NO_ROUND : tu + o0 - ran0, rest1 = sm1 == IDLE || fin1 ? NO_ROUND : tu + o1 - ran1;
          const unsigned fm0 = __ballot_sync(0xffffffffu, fin0), fm1 = __ballot_sync(0xffffffffu, fin1);
          const u32 rest = __reduce_min_sync(0xffffffffu, min(rest0, rest1));
          if (lane == 0) first_fin[b] = rest;
          nc = min(nc, rest);
          if (!(fm0 | fm1)) continue;
          if (__popc(fm0) + __popc(fm1) == 1) {         // one run
            const u32 j = __shfl_sync(0xffffffffu, fm0 ? j0 : j1, __ffs(static_cast<int>(fm0 | fm1)) - 1), so = lengths[j], o = so >> 16;
            if (lane == 0) {
              done[j >> 5] |= 1u << (j & 31u);
              sst[j] = static_cast<unsigned short>(IDLE);
              if (KVS_OK_AT(j, n, CHK_SP_JOB)) { js[j] = t - static_cast<int>(o); jc[j] = t; }
              steps += o; flow += t; ++runs; hmax = max(hmax, t);
            }
            A -= (so & 0xffffu) + 1u - (tu - o);
            --cnt; --left;
          } else {
            u32 dA = 0, n_fin = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const u32 j = h ? j1 : j0, so = h ? so1 : so0, o = so >> 16;
              if ((h ? fin1 : fin0) && (atomicOr(&done[j >> 5], 1u << (j & 31u)) >> (j & 31u) & 1u) == 0) {   // the first of its entries
                sst[j] = static_cast<unsigned short>(IDLE);
                if (KVS_OK_AT(j, n, CHK_SP_JOB)) { js[j] = t - static_cast<int>(o); jc[j] = t; }
                steps += o; flow += t; ++runs; hmax = max(hmax, t);
                dA += (so & 0xffffu) + 1u - (tu - o);
                ++n_fin;
              }
            }
            const int kf = static_cast<int>(__reduce_add_sync(0xffffffffu, n_fin));
            A -= __reduce_add_sync(0xffffffffu, dA);
            cnt -= kf; left -= kf;
          }
          __syncwarp();
        }
      }
      next_comp = __reduce_min_sync(0xffffffffu, nc);
      __syncwarp();
    }
    // slots that have ended: a job killed at the end of its slot is free again
    if (ne <= t) {
      const int eend = ph.ahead ? 0 : ph.started(t - static_cast<int>(ph.tau) - ph.base);
      do {
        bool act;
        if (ph.ahead) {
          act = (end_mask >> lane & 1u) != 0 && end_at <= t;
          end_mask &= ~__ballot_sync(0xffffffffu, act);
        } else {
          const int r = re + lane;
          act = r < eend;
          end_job = act ? job_of(r) : 0u;
          re = min(re + 32, eend);
        }
        const bool fr = act && !is_done(end_job);
        if (fr) atomicOr(&free_map[end_job >> 5], 1u << (end_job & 31u));
        const unsigned hit = __ballot_sync(0xffffffffu, fr);
        if (hit) {                                      // ranks are in index order
          const int j = static_cast<int>(__shfl_sync(0xffffffffu, end_job, __ffs(static_cast<int>(hit)) - 1));
          freed(j, lengths[j] & 0xffffu);
        }
        if (ph.ahead) {
          if (end_mask) ne = __shfl_sync(0xffffffffu, end_at, __ffs(static_cast<int>(end_mask)) - 1);
          else next_ends();
        } else if (re >= eend) {
          ne = re < ph.np ? ph.start_of(re) + static_cast<int>(ph.tau) : NEVER;
        }
      } while (ne <= t);
      __syncwarp();
    }
    // the next phase begins: its participants are the jobs of a later class, in index order
    if (t == phase_at) {
      int kept = 0;
      for (int q0 = 0; q0 < ph.np; q0 += 32) {
        const int q = q0 + lane;
        const u32 j = q < ph.np ? job_of(q) : 0u;
        const bool keep = q < ph.np && lengths[j] >> 16 > ph.tau;
        const unsigned km = __ballot_sync(0xffffffffu, keep);
        __syncwarp();
        const int d = kept + __popc(km & lt_mask);
        if (keep && KVS_OK_AT(d, n, CHK_SP_LIST)) list[d] = static_cast<unsigned short>(j);
        kept += __popc(km);
        __syncwarp();
      }
      ++phase;
      all_take_part = kept == n;
      enter(phase, kept);
      rs = 0; re = 0; ns = ph.base; ne = ph.base + static_cast<int>(ph.tau);
      phase_at = phase + 1 < L && sh.np[phase + 1] > 0 ? sh.pbase[phase + 1] : NEVER;
      if (ph.ahead) { look_ahead(w, t, false); apply_ring(w, 0u, 0u); }
    }
    // (2) pipeline runs that start now
    if (ns <= t) {
      const int rend = ph.ahead ? 0 : ph.started(t - ph.base);
      do {
        unsigned acting;
        if (ph.ahead) {
          acting = __ballot_sync(0xffffffffu, (start_mask >> lane & 1u) != 0 && start_at <= t);
          start_mask &= ~acting;
        } else {                                        // ranks [rs, rend), 32 at a time (they concern different jobs)
          const int r = rs + lane;
          start_job = r < rend ? job_of(r) : 0u;
          const u32 so = lengths[start_job];
          start_o = so >> 16; start_s1 = (so & 0xffffu) + 1u;
          acting = __ballot_sync(0xffffffffu, r < rend);
          rs = min(rs + 32, rend);
        }
        if ((acting & (acting - 1u)) == 0) {            // one run: no votes and no sums over lanes
          const int src = __ffs(static_cast<int>(acting)) - 1;
          const u32 j = __shfl_sync(0xffffffffu, start_job, src), o = __shfl_sync(0xffffffffu, start_o, src), s1 = __shfl_sync(0xffffffffu, start_s1, src);
          const u32 sm = sst[j], len = min(o, ph.tau);
          const int end = t + static_cast<int>(len);
          if (is_done(j)) {                             // dropped from the plan
            drop_now(w, t, s1 - tu, 1u, end);
          } else {
            const bool comp = len == o;
            if (sm != IDLE) {                           // its speculative run is killed; the stack entry goes stale
              const u32 ran = running_for(sm);
              A -= s1 - (tu - ran);
              --cnt;
              if (lane == 0) { steps += ran; runs += ran > 0 ? 1u : 0u; }
            }
            __syncwarp();
            if (lane == 0) {
              steps += len; ++runs;
              sst[j] = static_cast<unsigned short>(IDLE);
              free_map[j >> 5] &= ~(1u << (j & 31u));
              if (comp) {
                done[j >> 5] |= 1u << (j & 31u);
                if (KVS_OK_AT(j, n, CHK_SP_JOB)) { js[j] = t; jc[j] = end; }
                flow += end;
                hmax = max(hmax, end);
              }
            }
            left -= comp ? 1 : 0;
            if (static_cast<int>(j) == cj) cj = -1;
          }
          __syncwarp();
        } else {
          const bool act = (acting >> lane & 1u) != 0;
          const u32 j = act ? start_job : 0u, o = start_o, s1 = start_s1, sm = sst[j], len = min(o, ph.tau);
          const bool dn = is_done(j), run = act && !dn, drop = act && dn, comp = run && len == o;
          const bool kill = run && sm != IDLE;
          const unsigned km = __ballot_sync(0xffffffffu, kill), dm = __ballot_sync(0xffffffffu, drop), cm = __ballot_sync(0xffffffffu, comp);
          if (__any_sync(0xffffffffu, run && static_cast<int>(j) == cj)) cj = -1;
          left -= __popc(cm);
          if (km) {
            const u32 ran = running_for(sm);
            A -= __reduce_add_sync(0xffffffffu, kill ? s1 - (tu - ran) : 0u);
            cnt -= __popc(km);
            if (kill) { steps += ran; runs += ran > 0 ? 1u : 0u; }
          }
          if (run) {
            steps += len; ++runs;
            sst[j] = static_cast<unsigned short>(IDLE);
            if (!kill) atomicAnd(&free_map[j >> 5], ~(1u << (j & 31u)));
          }
          if (comp) {
            atomicOr(&done[j >> 5], 1u << (j & 31u));
            if (KVS_OK_AT(j, n, CHK_SP_JOB)) { js[j] = t; jc[j] = t + static_cast<int>(len); }
            flow += t + static_cast<int>(len);
            hmax = max(hmax, t + static_cast<int>(len));
          }
          // dropped from the plan: those that would have held their whole slot together, those that reach beyond the window
          // together, the others one by one
          if (dm) {
            const int end = t + static_cast<int>(len);
            const u32 v = s1 - tu;
            const unsigned wm = __ballot_sync(0xffffffffu, drop && len == ph.tau);
            if (wm) drop_now(w, t, __reduce_add_sync(0xffffffffu, drop && len == ph.tau ? v : 0u), static_cast<u32>(__popc(wm)), t + static_cast<int>(ph.tau));
            const bool rest = drop && len < ph.tau, beyond = rest && end >= w + 32 && end < w + ring_rounds;
            const unsigned bm = __ballot_sync(0xffffffffu, beyond);
            if (bm) {
              const u32 V = __reduce_add_sync(0xffffffffu, beyond ? v : 0u), c = static_cast<u32>(__popc(bm));
              if (w + lane >= t) Bw -= static_cast<int>(V + c * static_cast<u32>(w + lane));
              Ad += V; Cd += c;
              if (beyond) { atomicAdd(&ring_a[end & ring_mask], v); atomicAdd(&ring_c[end & ring_mask], 1u); }
            }
            unsigned om = __ballot_sync(0xffffffffu, rest && !beyond);
            while (om) {
              const int src = __ffs(static_cast<int>(om)) - 1;
              om &= om - 1u;
              const u32 vs = __shfl_sync(0xffffffffu, v, src);
              drop_now(w, t, vs, 1u, __shfl_sync(0xffffffffu, end, src));
            }
          }
          __syncwarp();
        }
        if (ph.ahead) {
          if (start_mask) ns = __shfl_sync(0xffffffffu, start_at, __ffs(static_cast<int>(start_mask)) - 1);
          else next_starts();
        } else if (rs >= rend) {
          ns = rs < ph.np ? ph.start_of(rs) : NEVER;
        }
      } while (ns <= t);
    }
    if (t == H) break;                                  // nothing runs in round H; only completions were due
    if (left == 0) {
      // Every job is done: what is left of the plan are the completing runs in progress (see k_spec)
      __threadfence();
      __syncwarp();
      const int first4 = t + static_cast<int>((4u - (reinterpret_cast<uintptr_t>(prof + t) >> 2 & 3u)) & 3u);
      for (int u = t + lane; u < min(first4, H); u += 32) prof[u] = 0;
      int last4 = first4;
      if (first4 + 4 <= H) last4 = first4 + ((H - first4) & ~3);
      for (int u = first4 + 4 * lane; u < last4; u += 128) *reinterpret_cast<int4*>(prof + u) = make_int4(0, 0, 0, 0);
      for (int u = last4 + lane; u < H; u += 32) prof[u] = 0;
      hmax = warp_max(hmax);
      __syncwarp();
      for (int r = ph.ahead ? end_first : re; r < rs; ++r) {
        const u32 j = job_of(r);
        const int end = jc[j];
        if (end > t && KVS_OK_AT(end, H + 1, CHK_SP_PROF)) {
          const int first = end - static_cast<int>(lengths[j] >> 16), sj = prompt(j);
          for (int u = t + lane; u < end; u += 32) prof[u] += sj + (u - first) + 1;
          __syncwarp();
        }
      }
      for (int u = t + lane; u < hmax; u += 32) peak = max(peak, static_cast<u32>(__ldcg(prof + u)));
      break;
    }
    const u32 B = static_cast<u32>(__shfl_sync(0xffffffffu, Bw, t & 31));
    // (3) the pipeline comes first
    while (cnt > 0 && B + A + tu * static_cast<u32>(cnt) > Mu) {
      u32 j = 0, sm = IDLE;
      while (top > 0 && sm == IDLE) {                   // the live entry nearest to the top: no other of its job is above it
        --top;
        j = KVS_OK_AT(top, m, CHK_SP_STACK) ? job_at(stk[top]) : 0u;
        sm = sst[j];
      }
      if (sm == IDLE) break;
      const u32 ran = running_for(sm), s0 = lengths[j] & 0xffffu;
      A -= s0 + 1u - (tu - ran);
      --cnt;
      steps += lane == 0 ? ran : 0u;
      runs += lane == 0 && ran > 0 ? 1u : 0u;
      __syncwarp();
      if (lane == 0) {
        sst[j] = static_cast<unsigned short>(IDLE);
        atomicOr(&free_map[j >> 5], 1u << (j & 31u));
      }
      __syncwarp();
      freed(static_cast<int>(j), s0);
    }
    // (4) first come first served: the lowest free job, and with it those of the 32 indices it lies among, as far as their
    // first rounds fit, in order; the first that does not fit ends the round's admissions
    for (;;) {
      const int room = static_cast<int>(Mu - (B + A + tu * static_cast<u32>(cnt)));
      if (cj == -2 || (cj >= 0 && cs + 1 > room) || room <= 0) break;
      if (cj == -1) {
        const int f = first_free();
        if (f < 0) { cj = -2; break; }
        cj = fj = static_cast<int>(job_at(static_cast<u32>(f)));
        cs = prompt(cj);
        if (cs + 1 > room) break;
      }
      const u32 j = (static_cast<u32>(cj) & ~31u) + lane, bits = free_map[j >> 5], so = lengths[j];
      const bool fr = (bits >> lane & 1u) != 0;
      const u32 s1 = fr ? (so & 0xffffu) + 1u : 0u;
      u32 need = __reduce_add_sync(0xffffffffu, s1);    // below 32 * 2^16
      if (need > static_cast<u32>(room)) {              // inclusive sums, in index order
        need = s1;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const u32 y = __shfl_up_sync(0xffffffffu, need, d);
          if (lane >= d) need += y;
        }
      }
      const bool ok = fr && need <= static_cast<u32>(room);
      const unsigned okm = __ballot_sync(0xffffffffu, ok);    // the lowest free job at least
      const int got = __popc(okm);
      if (top + 32 > m || top > 3 * cnt + 256) purge(t);
      const u32 fin = ok ? tu + (so >> 16) : NO_ROUND;
      if (ok) {
        const int d = top + __popc(okm & lt_mask);
        if (KVS_OK_AT(d, m, CHK_SP_STACK) && KVS_OK_AT(j, n, CHK_SP_JOB)) {
          sst[j] = static_cast<unsigned short>(tm);
          stk[d] = static_cast<unsigned short>(j);
          js[j] = d;
          atomicMin(&first_fin[d / STK_BLK], fin);
        }
      }
      if (lane == 0) free_map[j >> 5] = bits & ~okm;
      A += __reduce_add_sync(0xffffffffu, ok ? s1 - tu : 0u);
      top += got;
      cnt += got;
      next_comp = min(next_comp, __reduce_min_sync(0xffffffffu, fin));
      const unsigned failed = bits & ~okm;
      __syncwarp();
      if (failed) {                                     // the first free job that does not fit is the candidate from now on
        const int src = __ffs(static_cast<int>(failed)) - 1;
        cj = fj = (cj & ~31) + src;
        cs = static_cast<int>(__shfl_sync(0xffffffffu, s1, src)) - 1;
        break;
      }
      fj = (cj & ~31) + 32;
      cj = -1;
    }
    if (cnt == 0) top = 0;                              // only stale entries are left
    // (5) the memory of this round, and of those up to the next event in which nothing can happen
    {
      const int stop = static_cast<int>(min(static_cast<u32>(min(min(min(ns, ne), phase_at), min(w + 32, H))), next_comp));
      const int u = w + lane;
      const u32 mem = static_cast<u32>(Bw) + A + static_cast<u32>(u) * static_cast<u32>(cnt);
      const int room = static_cast<int>(Mu - mem);
      const bool quiet = !(cnt > 0 && room < 0) && (cj == -2 || room <= 0 || (cj >= 0 && cs + 1 > room));
      const unsigned busy = __ballot_sync(0xffffffffu, u > t && u < stop && !quiet);
      const int next = max(t + 1, busy ? w + __ffs(static_cast<int>(busy)) - 1 : stop);
      if (u >= t && u < next) {
        if (KVS_OK_AT(u, H, CHK_SP_PROF)) prof[u] = static_cast<int32_t>(mem);
        peak = max(peak, mem);
      }
      tm += static_cast<u32>(next - t);
      if (tm >= MODT) tm -= MODT;
      t = next;
    }
  }
  flow = warp_sum(flow); steps = warp_sum(steps); runs = __reduce_add_sync(0xffffffffu, runs); peak = __reduce_max_sync(0xffffffffu, peak);
  hmax = warp_max(hmax);
  if (lane == 0) {
    if (p.peak) p.peak[e] = peak;
    if (p.flow) p.flow[e] = flow;
    if (p.job_steps) p.job_steps[e] = steps;
    if (p.n_runs) p.n_runs[e] = runs;
    if (p.n_unfinished) p.n_unfinished[e] = left;
    p.horizon[e] = hmax;
    if (p.feasible) p.feasible[e] = peak <= Mu ? 1 : 0;
  }
}

}  // namespace

KVS_DEFINE_CHECK_WORD(kvs_spec_check_word)

i64 kvs_spec_warp_bytes(i64 max_jobs) { return spec_stride(max_jobs); }

// Once per device, before the first launch.
cudaError_t kvs_setup_spec() { return cudaFuncSetAttribute(k_spec_smem, cudaFuncAttributeMaxDynamicSharedMemorySize, SPEC_SMEM); }

// The on-chip kernel over p.groups, if there are any, and the other one over what it has left (or over the whole list).
cudaError_t kvs_launch_spec(SpecParams p, cudaStream_t stream) {
  if (p.n_list <= 0 || p.n_warps <= 0) return cudaSuccess;
  if (p.n_groups > 0) {
    const int n = static_cast<int>(p.max_jobs);
    k_spec_smem<<<static_cast<unsigned>(p.n_groups), 32 * p.group_warps, spec_cta_bytes(n, p.group_warps, p.ring), stream>>>(p, n, p.ring);
  } else {
    p.left_list = nullptr;
  }
  k_spec<<<static_cast<unsigned>((p.n_warps + SWARPS - 1) / SWARPS), ST, 0, stream>>>(p);
  return cudaGetLastError();
}
