// Bounds on total flow time that depend on an instance only through its class sizes
// (Lemma "Area-Based Lower Bound for OPT", Lemma "GBA Upper Bound via Packing Efficiency",
// Lemma "GSA Upper Bound via Packing Efficiency").
//
// Per (instance, setting): the ladder tau_p with k_p = k*(tau_p, s_bar) and the sizes of the classes of the response
// lengths (class = first p with tau_p >= o); then, by one warp with a lane per phase, in exact integers (128 bits where
// 64 do not do)
//   ladder term        Q_p = n_p tau_p + sum_{i < n_p} floor(i tau_p / k_p)   (closed form: floor sum)
//   class-prefix term  S_p = sum_{q < p} (floor(n_q tau_q / k_q) + tau_q)
//   UpperGBA           = sum_p (n_p S_p + Q_p)
//   spillover cost     D_p = ceil(n_{>p} tau_p / k_p)
//   phase-prefix cost  T_p = sum_{q < p} (floor(n_{>=q} tau_q / k_q) + tau_q)
//   GSA bound          = sum_p n_p (T_p + D_p) + sum_p Q_p
//   2 M * lower bound  = sum_p 2 Area(x_p, s_bar) (n_p (n_p + 1) / 2 + n_{>p} n_p),
//                        Area(x, s) = s x + x (x + 1) / 2, x_0 = 0 and x_p = tau_(p-1): every job of
//                        class p is longer than x_p (the integer part of the paper's real threshold).
//
// What bounds it: the shared-memory work of one histogram per instance and the latency of the phases' divisions, not the
// one pass over s and o.  8,192 evaluations (1,024 instances of 10,000 jobs, eight settings each): one thread per evaluation
// adding the phases up in 128-bit divisions 765 us; a lane per phase in the same kernel 348 us (102 registers left two
// CTAs per SM to hide the chain); as two kernels 133 us for a histogram per evaluation and 36 us for the sums; with one
// histogram per instance (k_class_counts) 56 us and 36 us.
#include "kvs_events.cuh"
#include "kvs_ladder.cuh"

namespace {

constexpr int BW = 4;         // evaluations (warps) per CTA of the second kernel
constexpr int MAXP = KVS_MAX_PHASES;

struct Ladder {
  u128 pw_a[MAXP + 1];
  u128 pw_b[MAXP + 1];
  u32 tau[MAXP], k[MAXP];
  int n_phases;
};

__device__ __forceinline__ u128 shfl_up128(u128 v, int d) {
  const u64 lo = __shfl_up_sync(0xffffffffu, static_cast<u64>(v), d), hi = __shfl_up_sync(0xffffffffu, static_cast<u64>(v >> 64), d);
  return static_cast<u128>(hi) << 64 | lo;
}
__device__ __forceinline__ u128 bcast128(u128 v, int src) {
  const u64 lo = __shfl_sync(0xffffffffu, static_cast<u64>(v), src), hi = __shfl_sync(0xffffffffu, static_cast<u64>(v >> 64), src);
  return static_cast<u128>(hi) << 64 | lo;
}
// exclusive sum over the lanes; *total = the sum over all of them
__device__ __forceinline__ u128 excl128(u128 v, u128* total) {
  u128 incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const u128 y = shfl_up128(incl, d);
    if (static_cast<int>(lane_id()) >= d) incl += y;
  }
  *total = bcast128(incl, 31);
  return incl - v;
}

// What both kernels derive from a setting; status 0 = the bounds are defined.
struct Case {
  i64 lo, s_bar, M, X;
  int n, status;
};
__device__ __forceinline__ Case case_of(const i64* job_off, const InstStats& is, const kvs_setting& st) {
  Case c;
  c.lo = job_off[st.instance];
  c.n = is.flags ? 0 : static_cast<int>(job_off[st.instance + 1] - c.lo);
  c.M = st.M;
  c.s_bar = st.s_bar >= 0 ? st.s_bar : is.s_max;
  c.X = c.M - c.s_bar;
  c.status = is.flags;
  if (!c.status && (c.X < 1 || is.o_max > c.X)) c.status = KVS_EVAL_INFEASIBLE;
  return c;
}

// tau_p = X >> (L - 1 - p), L the bit length of X
__device__ __forceinline__ bool is_pow2(const kvs_setting& st) { return st.alpha_num == 2 && st.alpha_den == 1 && st.beta0 <= 0; }

// Statistics of the instances and jobs per class of every evaluation: counts[e * MAXP + p].  One CTA per run of evaluations
// of one instance (runs[2 r] = first evaluation, runs[2 r + 1] = how many).  A setting's class sizes are differences of the
// cumulative counts of o at its slices, so one histogram over the values of o serves all settings of the run: the jobs
// are read and counted once, not once per setting.  Responses of BINS and more go through class_of per setting.
constexpr int BINS = 16512;                                 // 64.5 KB of shared memory: three CTAs per SM
constexpr int BT = 512;
constexpr int BIN_PER = BINS / BT + 1;                      // bins per thread of the scan: odd, no bank conflicts
__global__ void __launch_bounds__(BT, 3) k_class_counts(const i64* __restrict__ job_off, const int32_t* __restrict__ s, const int32_t* __restrict__ o, i64 max_jobs,
                                                        InstStats* __restrict__ stats, const __grid_constant__ BoundSettings settings,
                                                        const i64* __restrict__ runs, u32* __restrict__ counts) {
  extern __shared__ u32 bin[];                              // BIN_PER * BT words
  __shared__ Ladder sh;
  __shared__ u32 cnt[MAXP];
  __shared__ int red[32];
  __shared__ u32 wsum[32];
  __shared__ kvs_setting sts[BT / 32];
  const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  const i64 e0 = runs[2 * static_cast<i64>(blockIdx.x)], n_e = runs[2 * static_cast<i64>(blockIdx.x) + 1];
  // the settings lie in page-locked host memory (a read takes microseconds): one per warp, all of them together
  constexpr int SW = sizeof(kvs_setting) / 4;
  auto fetch = [&](i64 first) {
    const int n_sets = static_cast<int>(min_i64(BT / 32, e0 + n_e - first)), n_words = n_sets * SW;
    if (settings.brief) { if (tid < n_sets) sts[tid] = settings[first + tid]; }
    else for (int i = tid; i < n_words; i += BT) reinterpret_cast<u32*>(sts)[i] = reinterpret_cast<const u32*>(settings.full + first)[i];
  };
  fetch(e0);
  __syncthreads();
  const i64 inst = sts[0].instance;
  const i64 lo = job_off[inst], hi = job_off[inst + 1];
  int flags = (hi < lo || hi - lo > max_jobs) ? KVS_EVAL_BAD_INPUT : 0;
  const int n = flags ? 0 : static_cast<int>(hi - lo);
  for (int i = tid; i < BIN_PER * BT; i += BT) bin[i] = 0;
  __syncthreads();
  int s_max = 0, o_max = 0, bad = 0;
  constexpr int U = 4;                                      // loads in flight per thread
  for (int j0 = tid; j0 < n; j0 += U * BT) {
    int sv[U], ov[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + u * BT;
      sv[u] = j < n ? __ldg(s + lo + j) : 0;
      ov[u] = j < n ? __ldg(o + lo + j) : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j0 + u * BT >= n) continue;
      s_max = max(s_max, sv[u]); o_max = max(o_max, ov[u]);
      bad |= (sv[u] < 0) | (ov[u] < 1);
      if (static_cast<u32>(ov[u]) < static_cast<u32>(BINS)) atomicAdd(&bin[ov[u]], 1u);
    }
  }
  s_max = block_max(s_max, red, 0);
  o_max = block_max(o_max, red, 0);
  bad = block_max(bad, red, 0);
  if (bad) flags = KVS_EVAL_BAD_INPUT;
  const InstStats is{s_max, o_max, o_max, flags};
  if (tid == 0) stats[inst] = is;
  // cumulative counts: bin[v] = jobs with o <= v (block_max has synchronised the histogram)
  u32 sum = 0;
#pragma unroll 1
  for (int i = 0; i < BIN_PER; ++i) { sum += bin[tid * BIN_PER + i]; bin[tid * BIN_PER + i] = sum; }
  const u32 incl = warp_incl(sum);
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  u32 before = incl - sum;
  for (int w = 0; w < warp; ++w) before += wsum[w];
  if (before)
    for (int i = 0; i < BIN_PER; ++i) bin[tid * BIN_PER + i] += before;
  __syncthreads();
  for (i64 first = e0; first < e0 + n_e; first += BT / 32) {
    if (first != e0) { fetch(first); __syncthreads(); }
    const int m = static_cast<int>(min_i64(BT / 32, e0 + n_e - first));
    if (warp < m) {                                         // alpha = 2, every response in the histogram: one warp per setting
      const kvs_setting& st = sts[warp];
      const Case c = case_of(job_off, is, st);
      if (!c.status && is_pow2(st) && o_max < BINS) {
        const u32 Xc = static_cast<u32>(c.X);
        const int L = 32 - __clz(Xc);
        if (lane < L) {
          const u32 t = Xc >> (L - 1 - lane), t0 = lane == 0 ? 0u : Xc >> (L - lane);
          counts[(first + warp) * MAXP + lane] = bin[min(t, static_cast<u32>(BINS - 1))] - bin[min(t0, static_cast<u32>(BINS - 1))];
        }
      }
    }
    for (int x = 0; x < m; ++x) {                           // the others by the whole block
      const kvs_setting& st = sts[x];
      const Case c = case_of(job_off, is, st);
      if (c.status || (is_pow2(st) && o_max < BINS)) continue;
      const i64 e = first + x;
      if (tid < 32) ladder_phases(sh, c.X, st.alpha_num, st.alpha_den, st.beta0, [](u32) { return 0u; });
      for (int i = tid; i < MAXP; i += BT) cnt[i] = 0;
      __syncthreads();
      const int L = sh.n_phases;                            // 0: more phases than the tables hold
      if (o_max < BINS) {
        for (int q = tid; q < L; q += BT)
          counts[e * MAXP + q] = bin[min(sh.tau[q], static_cast<u32>(BINS - 1))] - (q ? bin[min(sh.tau[q - 1], static_cast<u32>(BINS - 1))] : 0u);
      } else {
        for (int j = tid; j < n && L > 0; j += BT) atomicAdd(&cnt[class_of(sh.tau, L, static_cast<u32>(__ldg(o + lo + j)))], 1u);
        __syncthreads();
        for (int q = tid; q < L; q += BT) counts[e * MAXP + q] = cnt[q];
      }
      __syncthreads();                                      // the next setting writes the tables again
    }
    __syncthreads();                                        // every warp has read these settings before the next are fetched
  }
}

// The sums over the phases, one warp per evaluation, one lane per phase.
__global__ void __launch_bounds__(BW * 32) k_bounds(const i64* __restrict__ job_off, const InstStats* __restrict__ stats,
                                                    const __grid_constant__ BoundSettings settings, i64 P, const u32* __restrict__ counts,
                                                    kvs_bounds_out out) {
  __shared__ Ladder shs[BW];
  const int lane = lane_id();
  Ladder& sh = shs[threadIdx.x >> 5];
  const i64 e = static_cast<i64>(blockIdx.x) * BW + (threadIdx.x >> 5);
  if (e >= P) return;
  const kvs_setting st = settings[e];
  const Case c = case_of(job_off, stats[st.instance], st);
  int status = c.status;
  if (!status) {
    ladder32(sh, c.X, st.alpha_num, st.alpha_den, st.beta0, static_cast<u32>(c.s_bar), static_cast<u32>(c.M));
    if (sh.n_phases == 0) status = KVS_EVAL_RANGE;
  }
  u128 upper_gba = 0, gsa = 0, lower = 0;
  if (!status) {
    const int L = sh.n_phases;
    const u128 LIMIT = (static_cast<u128>(1) << 63) - 1;
    u128 class_prefix = 0, phase_prefix = 0, before = 0;  // sums over the phases of earlier groups of 32
    for (int p0 = 0; p0 < L; p0 += 32) {
      const int p = p0 + lane;
      const bool on = p < L;
      const u64 np = on ? counts[e * MAXP + p] : 0, t = on ? sh.tau[p] : 0, kk = on ? sh.k[p] : 1;
      u128 tot_n, tot_c, tot_g;
      const u64 n_lt = static_cast<u64>(before + excl128(np, &tot_n));
      const u64 n_ge = static_cast<u64>(c.n) - n_lt, n_gt = n_ge - np;
      u64 qc, qg, qd, r;
      divmod_u(np * t, kk, &qc, &r);                       // every product here is below 2^62
      divmod_u(n_ge * t, kk, &qg, &r);
      divmod_u(n_gt * t + kk - 1, kk, &qd, &r);
      const u128 S = class_prefix + excl128(on ? static_cast<u128>(qc) + t : 0, &tot_c);
      const u128 Tp = phase_prefix + excl128(on ? static_cast<u128>(qg) + t : 0, &tot_g);
      const u128 Q = static_cast<u128>(np) * t + (np ? floor_sum<u128>(np, kk, t, 0) : 0);
      const u64 x = p == 0 || !on ? 0 : sh.tau[p - 1];
      const u128 area2 = static_cast<u128>(2) * static_cast<u64>(c.s_bar) * x + static_cast<u128>(x) * (x + 1);
      const u128 a = on ? static_cast<u128>(np) * S + Q : 0, b = on ? static_cast<u128>(np) * (Tp + qd) + Q : 0;
      const u128 d = on ? area2 * (static_cast<u128>(np) * (np + 1) / 2 + static_cast<u128>(n_gt) * np) : 0;
      u128 ta, tb, td;
      excl128(a, &ta); excl128(b, &tb); excl128(d, &td);
      upper_gba += ta; gsa += tb; lower += td;
      before += tot_n; class_prefix += tot_c; phase_prefix += tot_g;
    }
    // the terms are non-negative, so a partial sum beyond the limit shows in the total
    if (upper_gba > LIMIT || gsa > LIMIT || lower > LIMIT) status = KVS_EVAL_RANGE;
  }
  if (lane == 0) {
    const bool ok = status == 0;
    if (out.upper_gba) out.upper_gba[e] = ok ? static_cast<i64>(upper_gba) : -1;
    if (out.upper_gsa) out.upper_gsa[e] = ok ? static_cast<i64>(gsa) : -1;
    if (out.lower_2m) out.lower_2m[e] = ok ? static_cast<i64>(lower) : -1;
    if (out.status) out.status[e] = status;
  }
}

}  // namespace

// Once per device, before the first launch.
cudaError_t kvs_setup_bounds() {
  return cudaFuncSetAttribute(k_class_counts, cudaFuncAttributeMaxDynamicSharedMemorySize, BIN_PER * BT * 4);
}

// runs: n_runs pairs (first evaluation, number of evaluations) of evaluations of one instance; counts: P * KVS_MAX_PHASES words
cudaError_t kvs_launch_bounds(const i64* job_off, const int32_t* s, const int32_t* o, i64 max_jobs, InstStats* stats, const kvs_setting* list, i64 P,
                              const i64* runs, i64 n_runs, const kvs_bounds_out& out, u32* counts, cudaStream_t stream) {
  if (P <= 0) return cudaSuccess;
  const bool in_brief = list[0].family == KVS_SETTINGS_BRIEF;
  const BoundSettings settings{list, in_brief ? reinterpret_cast<const int2*>(list + 1) : nullptr, list[0]};
  k_class_counts<<<static_cast<unsigned>(n_runs), BT, BIN_PER * BT * 4, stream>>>(job_off, s, o, max_jobs, stats, settings, runs, counts);
  k_bounds<<<static_cast<unsigned>((P + BW - 1) / BW), BW * 32, 0, stream>>>(job_off, stats, settings, P, counts, out);
  return cudaGetLastError();
}
