// C ABI: argument validation, workspace layout, launches.  Host code only.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <functional>
#include <new>
#include <string>
#include <vector>

#include "kvs_internal.cuh"
#include "kvs_spec_shape.h"

constexpr int KVS_HOST_CHUNKS = 16;   // the host entry point pipelines copies and kernels over at most this many chunks
constexpr int KVS_CHUNK_EVALS = 512;  // of about this many evaluations
constexpr int KVS_LANES = 3;          // that take turns on this many pairs of streams, see open_side

struct kvs_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  unsigned char* workspace = nullptr;
  uint64_t workspace_bytes = 0;
  int sm_count = 0;
  int build_ctas_per_sm = 1;
  int fused_ctas_per_sm = 1;
  int light_ctas_per_sm = 1;
  bool timing = false;
  bool timed = false;
  bool split_timed = false;   // the last timed call took the fast path (event between its two variants)
  cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};   // before the ordering kernel, after it, after the last kernel, after the light variant
  // host entry point: input copies run on a stream of their own, one event per chunk of instances
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t chunk_ev[KVS_HOST_CHUNKS + 1] = {};
  // The full variant's kernels run on a stream beside the caller's, see open_side
  // (the full variant's of lane l at 2 l, that of the lane itself, in the host entry point, at 2 l + 1).
  struct Side { cudaStream_t stream = nullptr; cudaEvent_t from = nullptr, done = nullptr; bool open = false; } side[2 * KVS_LANES];
  // Page-locked staging for what a fused call uploads (settings, counters, evaluation lists): one copy per call that
  // leaves at once, instead of one pageable copy per array (the larger of which block the host).  Two slots in
  // turn: a call waits at most for the upload of the call before the last one.
  struct Stage { unsigned char* p = nullptr; size_t bytes = 0; cudaEvent_t done = nullptr; bool used = false; } stage[2];
  int next_stage = 0;
  bool fill = false;          // kvs_set_unwritten
  int32_t fill_job = 0, fill_prof = 0;
  void* pinned = nullptr;   // 256 bytes of page-locked memory for values that the host has to see
  std::string err;
};

// One caller's sizes on their way (kvs_sizes_begin, kvs_sizes_end).  Apart from the contexts: the wait for them is long, and another
// thread may use, or replace by a larger one, the context that the call will run on meanwhile.
struct kvs_reader {
  int device = 0;
  cudaStream_t stream = nullptr;                           // of the open request; the caller may destroy it when it never ends that
  struct Pinned { int64_t* p = nullptr; size_t bytes = 0; } in, rows;   // what is read: job offsets, then capacities; what goes up
  int64_t n_off = -1, n_cap = -1;                          // of the open request (-1: not asked for)
  bool open = false;
  cudaEvent_t arrived = nullptr;                           // the sizes of the open request
  cudaEvent_t sent = nullptr;                              // the rows of the last request have gone up
  bool sending = false;
  std::string err;
};

namespace {

constexpr int64_t KVS_MAX_GRID = 1024;        // upper bound on CTAs of the fused kernel (sizes the carry lists)
constexpr int64_t KVS_TIME_LIMIT = 1ll << 31; // exclusive bound on M, tau, k

// Nothing leaves a C entry point as an exception: host memory that runs out becomes a status (and, for the text of an error,
// an empty text).
template <class H, class F>
int guarded(H* handle, F body) noexcept {
  try {
    return body();
  } catch (...) {
    handle->err.clear();
    return KVS_E_STATE;
  }
}
template <class H>
int fail(H* handle, int code, const char* msg) {
  if (handle) guarded(handle, [&] { handle->err = msg; return 0; });
  return code;
}
template <class H>
int fail_cuda(H* handle, cudaError_t e, const char* where) {
  if (handle) guarded(handle, [&] { handle->err = std::string(where) + ": " + cudaGetErrorString(e); return 0; });
  return KVS_E_CUDA;
}

// A staging slot of at least `bytes` bytes whose last upload has finished.
cudaError_t take_stage(kvs_ctx* ctx, size_t bytes, kvs_ctx::Stage** out) {
  kvs_ctx::Stage& s = ctx->stage[ctx->next_stage];
  ctx->next_stage ^= 1;
  cudaError_t e = cudaSuccess;
  if (!s.done && (e = cudaEventCreateWithFlags(&s.done, cudaEventDisableTiming)) != cudaSuccess) return e;
  if (s.used && (e = cudaEventSynchronize(s.done)) != cudaSuccess) return e;
  if (s.bytes < bytes) {
    if (s.p) cudaFreeHost(s.p);
    s.p = nullptr; s.bytes = 0;
    const size_t want = bytes + bytes / 2 + 65536;
    if ((e = cudaMallocHost(reinterpret_cast<void**>(&s.p), want)) != cudaSuccess) return e;
    s.bytes = want;
  }
  *out = &s;
  return cudaSuccess;
}
// The slot is in use until the stream has got here.
cudaError_t mark_stage(kvs_ctx::Stage* s, cudaStream_t stream) {
  const cudaError_t e = cudaEventRecord(s->done, stream);
  s->used = e == cudaSuccess;
  if (e != cudaSuccess) cudaStreamSynchronize(stream);   // no event to wait for later
  return e;
}
// Uploads the first `bytes` bytes of the slot and marks it as in use until that has happened.
cudaError_t send_stage(kvs_ctx::Stage* s, void* dst, size_t bytes, cudaStream_t stream) {
  const cudaError_t e = cudaMemcpyAsync(dst, s->p, bytes, cudaMemcpyHostToDevice, stream);
  const cudaError_t marked = mark_stage(s, stream);
  return e != cudaSuccess ? e : marked;
}

size_t align_up(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

// Offsets of the scratch regions of the fused path inside the workspace.  Calls are ordered on
// one stream, so the entry points reuse the workspace from offset 0; the layout without staging
// is a prefix of the layout with staging.
struct Layout {
  size_t call;                                                          // what a call uploads, see call_bytes
  size_t stats, perm, perm_tmp, iperm, sorted_s, sorted_o, sorted_key, prefix_s, lists, fin_rank, slow_list;
  size_t class_counts;                                                  // of the bounds
  size_t sweep_unf, sweep_stat;                                         // unfinished counts and status words of a sweep over initial slices
  size_t st_off, st_s, st_o, st_key, st_arr;                            // host staging (inputs)
  size_t sc_peak, sc_flow, sc_steps, sc_hor, sc_unf, sc_feas, sc_stat;  // host staging (scalars)
  size_t total;
};

// What a fused call uploads in one piece: 256 bytes of work counters and list lengths, the settings, the list of
// evaluations of the full variant (which the light one appends to: P entries), the light variant's list, and the
// evaluations that the refill or speculative-run kernel works on afterwards.
// A call with few evaluations adds the sums of the evaluations that several CTAs share.
constexpr size_t CALL_COUNTERS = 256;
constexpr int KVS_RESIDENT_CTAS = 296;   // of the full variant on a B200: two per SM
constexpr int KVS_MAX_PARTS = 16;        // CTAs that share an evaluation (a ladder has 15 to 25 phases)

// CTAs per evaluation of a call with P evaluations of at most max_n jobs: as many as the GPU holds at a time.  Every CTA
// has scratch of its own, which for the largest instances would cost gigabytes: those are not shared.
int parts_for(int64_t P, int64_t max_n) {
  if (P < 1 || max_n > (1 << 18)) return 1;
  const int64_t g = KVS_RESIDENT_CTAS / P;
  return static_cast<int>(g < 1 ? 1 : (g > KVS_MAX_PARTS ? KVS_MAX_PARTS : g));
}
size_t lists_bytes(int64_t P) { return CALL_COUNTERS + static_cast<size_t>(P) * (sizeof(kvs_setting) + 3 * 8); }
size_t groups_at(int64_t P) { return lists_bytes(P) + static_cast<size_t>(P) * sizeof(FusedShare); }
size_t call_bytes(int64_t P) { return groups_at(P) + static_cast<size_t>(P) * 8 * KVS_SPEC_GROUP; }   // groups of evaluations of the speculative runs

Layout make_layout(int64_t N, int64_t I, int64_t max_n, int64_t P, bool staging) {
  Layout L{};
  size_t at = 0;
  auto take = [&](size_t bytes) { size_t r = at; at += align_up(bytes); return r; };
  L.call = take(call_bytes(P) + (KVS_HOST_CHUNKS + 1) * CALL_COUNTERS);   // the host entry point uploads chunk by chunk
  L.stats = take(static_cast<size_t>(I) * sizeof(InstStats));
  L.perm = take(static_cast<size_t>(N) * 4);
  L.perm_tmp = take(static_cast<size_t>(N) * 4);
  L.sorted_s = take(static_cast<size_t>(N) * 4);
  L.sorted_o = take(static_cast<size_t>(N) * 4);
  L.sorted_key = take(static_cast<size_t>(N) * 4);
  L.prefix_s = take(static_cast<size_t>(N + I) * 8);
  L.iperm = take(static_cast<size_t>(N) * 4);
  const int64_t grid = P < KVS_MAX_GRID ? P * parts_for(P, max_n) : KVS_MAX_GRID;
  L.lists = take(static_cast<size_t>(grid) * static_cast<size_t>(KVS_CTA_SCRATCH(max_n)));
  L.fin_rank = take(static_cast<size_t>(grid) * static_cast<size_t>(max_n) * 4);
  L.slow_list = take(static_cast<size_t>(P) * 8);
  L.class_counts = take(static_cast<size_t>(P) * KVS_MAX_PHASES * 4);
  L.sweep_unf = take(static_cast<size_t>(P) * 8);
  L.sweep_stat = take(static_cast<size_t>(P) * 4);
  if (staging) {
    L.st_off = take(static_cast<size_t>(I + 1) * 8);
    L.st_s = take(static_cast<size_t>(N) * 4);
    L.st_o = take(static_cast<size_t>(N) * 4);
    L.st_key = take(static_cast<size_t>(N) * 4);
    L.st_arr = take(static_cast<size_t>(N) * 8);
    L.sc_peak = take(static_cast<size_t>(P) * 8);
    L.sc_flow = take(static_cast<size_t>(P) * 8);
    L.sc_steps = take(static_cast<size_t>(P) * 8);
    L.sc_hor = take(static_cast<size_t>(P) * 8);
    L.sc_unf = take(static_cast<size_t>(P) * 8);
    L.sc_feas = take(static_cast<size_t>(P));
    L.sc_stat = take(static_cast<size_t>(P) * 4);
  }
  L.total = at;
  return L;
}

// Generic evaluator: per evaluation the tiled kernel's peak and count of finished tiles, the list of evaluations left to
// the 64-bit kernel, and its 64-bit constant terms and 32-bit slopes, capacity + one slot per evaluation.
struct GenericLayout { size_t peak, done, count, list, dconst, dcount, total; };
GenericLayout make_generic_layout(int64_t cap_total, int64_t P) {
  GenericLayout L{};
  size_t at = 0;
  auto take = [&](size_t bytes) { size_t r = at; at += align_up(bytes); return r; };
  L.peak = take(static_cast<size_t>(P) * 4);
  L.done = take(static_cast<size_t>(P) * 4);
  L.count = take(8);
  L.list = take(static_cast<size_t>(P) * 8);
  L.dconst = take(static_cast<size_t>(cap_total + P) * 8);
  L.dcount = take(static_cast<size_t>(cap_total + P) * 4);
  L.total = at;
  return L;
}

struct SweepLayout {
  size_t info, rec0, rec1, counts, part, sorted_s, sorted_o, prefix_s, prefix_s32, prefix_o, grid, table, total;
};

SweepLayout make_sweep_layout(int64_t max_n) {
  SweepLayout L{};
  size_t at = 0;
  auto take = [&](size_t bytes) { size_t r = at; at += align_up(bytes); return r; };
  const size_t n = static_cast<size_t>(max_n), chunks = static_cast<size_t>(kvs_order_chunks(max_n)) + 1;
  L.info = take(sizeof(OrderInfo));
  L.grid = take(2 * 65536 * 8 + 256);
  // the block maxima of the windows take the place of the records of the ordering
  const size_t table = static_cast<size_t>(KVS_SWEEP_TABLES) * static_cast<size_t>(kvs_sweep_blocks(max_n)) * 8;
  L.rec0 = L.table = take(std::max(table, 2 * align_up(n * 8)));
  L.rec1 = L.rec0 + align_up(n * 8);
  L.counts = take(chunks * 256 * 4);
  L.part = take(chunks * 16);
  L.sorted_s = take(n * 4);
  L.sorted_o = take(n * 4);
  L.prefix_s = take((n + 1) * 8);
  L.prefix_s32 = take((n + 1) * 4);
  L.prefix_o = take((n + 1) * 8);
  L.total = at;
  return L;
}

int check_instances(kvs_ctx* ctx, const kvs_instances* inst) {
  if (!inst) return fail(ctx, KVS_E_ARG, "instances: null");
  if (inst->n_instances < 0 || inst->n_jobs_total < 0 || inst->max_jobs_per_instance < 0)
    return fail(ctx, KVS_E_ARG, "instances: negative size");
  if (inst->max_jobs_per_instance >= (1ll << 31) - 1) return fail(ctx, KVS_E_RANGE, "instances: more than 2^31-2 jobs in one instance");
  if (!inst->job_off) return fail(ctx, KVS_E_ARG, "instances: job_off is null");
  if (inst->n_jobs_total > 0 && (!inst->s || !inst->o)) return fail(ctx, KVS_E_ARG, "instances: s or o is null");
  if (inst->window < 0) return fail(ctx, KVS_E_ARG, "instances: negative window");
  if (inst->window == 0 && inst->arrival) return fail(ctx, KVS_E_ARG, "instances: arrival given without a window (offline instances take arrival = NULL)");
  return KVS_OK;
}

// The ladder keeps a^j and X*b^j exactly in 128 bits.  With ell = floor(log_alpha X) the largest
// value formed is below a * X * b^(ell+1) (a^j <= X * b^j up to j = ell, one more factor for the
// test that ends the search); refuse parameters for which that might not fit, or that need more
// phases than the table holds.
bool ladder_fits(int64_t M, int a, int b) {
  const double la = std::log2(static_cast<double>(a)), lb = std::log2(static_cast<double>(b));
  const double lx = std::log2(static_cast<double>(M));
  const double ell = std::floor(lx / (la - lb)) + 1.0;   // one spare for rounding of the logarithms
  if (ell + 2.0 > KVS_MAX_PHASES) return false;
  return la + lx + (ell + 2.0) * lb < 125.0;             // also covers beta0 * a^p < a * X * b^p
}

// Whether what has been found right for setting b is right for a: they differ in nothing but the instance and the budget, which are
// looked at, and have the doubling ladder, whose length no budget makes too large.
bool like(const kvs_setting& a, const kvs_setting& b, int64_t n_instances) {
  return a.family == b.family && a.alpha_num == b.alpha_num && a.alpha_den == b.alpha_den && a.s_bar == b.s_bar && a.beta0 == b.beta0 &&
         a.tau == b.tau && a.k == b.k && a.subroutine == b.subroutine && a.per_class_s == b.per_class_s && a.alpha_num == 2 && a.alpha_den == 1 &&
         a.instance >= 0 && a.instance < n_instances && a.M >= 1 && a.M < KVS_TIME_LIMIT;
}

int check_settings(kvs_ctx* ctx, const kvs_instances* inst, const kvs_setting* st, int64_t P) {
  if (P < 0) return fail(ctx, KVS_E_ARG, "settings: negative count");
  if (P > 0 && !st) return fail(ctx, KVS_E_ARG, "settings: null");
  for (int64_t e = 0; e < P; ++e) {
    const kvs_setting& s = st[e];
    if (e > 0 && like(s, st[e - 1], inst->n_instances)) continue;
    if (s.instance < 0 || s.instance >= inst->n_instances) return fail(ctx, KVS_E_ARG, "settings: instance out of range");
    if (s.family < KVS_GBA || s.family > KVS_GSAS) return fail(ctx, KVS_E_ARG, "settings: unknown family");
    if (s.family == KVS_GSAS && (inst->o_est || inst->window != 0 || s.subroutine || s.per_class_s))
      return fail(ctx, KVS_E_ARG, "settings: speculative runs take offline instances without estimates and the plain slicing schedule");
    if (s.family == KVS_GBAD && (inst->o_est || inst->window != 0 || s.subroutine))
      return fail(ctx, KVS_E_ARG, "settings: the dynamic refill takes offline instances without estimates and the staggered subroutine");
    if (s.M < 1 || s.M >= KVS_TIME_LIMIT) return fail(ctx, KVS_E_RANGE, "settings: M outside [1, 2^31)");
    if (s.s_bar < -1) return fail(ctx, KVS_E_ARG, "settings: s_bar < -1");
    if (s.tau < 0 || s.tau >= KVS_TIME_LIMIT || s.k < 0 || s.k >= KVS_TIME_LIMIT)
      return fail(ctx, KVS_E_RANGE, "settings: tau or k outside [0, 2^31)");
    if (s.subroutine < 0 || s.subroutine > 1 || s.per_class_s < 0 || s.per_class_s > 1)
      return fail(ctx, KVS_E_ARG, "settings: subroutine and per_class_s are 0 or 1");
    if ((s.subroutine || s.per_class_s) && s.family != KVS_GBA && s.family != KVS_GSA && s.family != KVS_GBAD && s.family != KVS_GSAS)
      return fail(ctx, KVS_E_ARG, "settings: subroutine and per_class_s apply to the geometric families only");
    if (s.family == KVS_GBA || s.family == KVS_GSA || s.family == KVS_GBAD || s.family == KVS_GSAS) {
      if (s.alpha_den < 1 || s.alpha_num <= s.alpha_den) return fail(ctx, KVS_E_ARG, "settings: alpha must be > 1");
      if (s.beta0 < 0 || s.beta0 >= KVS_TIME_LIMIT) return fail(ctx, KVS_E_RANGE, "settings: beta0 outside [0, 2^31)");
      if (!(s.alpha_num == 2 && s.alpha_den == 1) && !ladder_fits(s.M, s.alpha_num, s.alpha_den))
        return fail(ctx, KVS_E_RANGE, "settings: ladder for this alpha and M needs more than 96 phases or 128-bit integers");
    }
  }
  return KVS_OK;
}

// Sorts numbers that lie in the lowest `bits` bits by what is above them (stable), eleven bits at a time; digits that all of them share
// cost one look.  2,048 evaluations of two families and eight budgets: 15 us, 110 with a comparison sort of the settings.
void sort_above(std::vector<uint64_t>& v, int bits) {
  if (v.size() < 64) { std::sort(v.begin(), v.end()); return; }         // the numbers themselves are in order
  uint64_t any = 0, all = ~0ull;
  for (uint64_t x : v) { any |= x; all &= x; }
  const uint64_t differ = any ^ all;
  std::vector<uint64_t> other(v.size());
  for (int at = bits; at < 64; at += 11) {
    if (((differ >> at) & 2047u) == 0) continue;
    size_t start[2049] = {};
    for (uint64_t x : v) ++start[((x >> at) & 2047u) + 1];
    for (int d = 0; d < 2048; ++d) start[d + 1] += start[d];
    for (uint64_t x : v) other[start[(x >> at) & 2047u]++] = x;
    v.swap(other);
  }
}

// The kernels of a call that is split by family do not depend on one another, and each of them ends with SMs that wait for
// its last evaluations.  So the full variant's run on a stream of their own, of higher priority (their evaluations are the
// longer ones), and the light variant's fill the places they leave.  The host entry point has its chunks of instances take
// turns on KVS_LANES such pairs of streams, each with CTA scratch of its own: a chunk's ordering, which leaves most of the GPU
// idle, and its last evaluations run beside the chunks before and after it (1,024 instances of up to 20,000 jobs, four
// families, in chunks of 512 evaluations: 3.63 ms with three lanes, 4.05 with two, 6.0 with every kernel on one stream).
// Opened behind what `from` holds; closing makes `to` wait.
cudaError_t open_side(kvs_ctx::Side& sd, cudaStream_t from, bool urgent) {
  cudaError_t e = cudaSuccess;
  int least = 0, greatest = 0;
  if (!sd.stream && ((e = cudaDeviceGetStreamPriorityRange(&least, &greatest)) != cudaSuccess ||
                     (e = cudaStreamCreateWithPriority(&sd.stream, cudaStreamNonBlocking, urgent ? greatest : least)) != cudaSuccess))
    return e;
  for (cudaEvent_t* ev : {&sd.from, &sd.done})
    if (!*ev && (e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming)) != cudaSuccess) return e;
  if ((e = cudaEventRecord(sd.from, from)) != cudaSuccess) return e;
  sd.open = true;
  return cudaStreamWaitEvent(sd.stream, sd.from, 0);
}
cudaError_t close_side(kvs_ctx::Side& sd, cudaStream_t to) {
  if (!sd.open) return cudaSuccess;
  cudaError_t e = cudaEventRecord(sd.done, sd.stream);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(to, sd.done, 0);
  if (e != cudaSuccess) e = cudaStreamSynchronize(sd.stream);   // the events failed: wait here
  if (e == cudaSuccess) sd.open = false;
  return e;
}
cudaError_t close_sides(kvs_ctx* ctx) {
  cudaError_t e = cudaSuccess;
  for (kvs_ctx::Side& sd : ctx->side) {
    const cudaError_t x = close_side(sd, ctx->stream);
    if (e == cudaSuccess) e = x;
  }
  return e;
}

// A call on a sub-range of the instances (host entry point): the `P` settings all name instances in
// [i0, i1) and are evaluations e0 .. e0 + P - 1 of a batch of P_total; `ev` already points at e0.  What chunk
// number `chunk` uploads goes to the copy stream before the chunk's inputs (behind them it would wait in the copy
// engine for the inputs of the chunks that follow); `feed` then sends the inputs and makes the kernels' stream wait.
// `lane`: the pair of streams that the chunk's kernels run on, or -1 for the context's stream; `light_ctas`: see lane_light_ctas.
struct FusedRange { int64_t i0, i1, e0, P_total; int chunk, lane; int64_t light_ctas; std::function<int()> feed; };

// CTA scratch of a lane, and the part of it at its start that the light variant's kernels take where the full variant's run
// beside them.  That part is the same for all chunks of a call: a lane's stream does not wait for its side stream between two
// chunks, so the light kernels of one run while the full kernels of the one before it may still use theirs.
constexpr int64_t LANE_CTAS = KVS_MAX_GRID / KVS_LANES;
int64_t lane_light_ctas(const kvs_setting* st, int64_t P) {
  for (int64_t e = 0; e < P; ++e)
    if (st[e].family != KVS_GSA) return LANE_CTAS / 2;
  return 0;                                  // no evaluation of the light variant (no profile is stored here)
}

int enqueue_fused(kvs_ctx* ctx, const kvs_instances* inst, const kvs_setting* settings, int64_t P,
                  const kvs_schedule_out* out, const kvs_eval_out* ev, int do_profile, const FusedRange* rg) {
  int rc = check_instances(ctx, inst);
  if (rc) return rc;
  rc = check_settings(ctx, inst, settings, P);
  if (rc) return rc;
  kvs_schedule_out o{};
  kvs_eval_out v{};
  if (out) o = *out;
  if (ev) v = *ev;
  const bool job_out = o.job_start || o.job_completion || o.job_start64 || o.job_completion64;
  if (job_out && !o.job_out_off) return fail(ctx, KVS_E_ARG, "schedule_out: job outputs need job_out_off");
  const bool run_out = o.run_job || o.run_phase || o.run_start || o.run_len || o.run_s;
  if (run_out && !o.run_off) return fail(ctx, KVS_E_ARG, "schedule_out: run outputs need run_off");
  if (v.profile && !v.profile_off) return fail(ctx, KVS_E_ARG, "eval_out: profile needs profile_off");
  if (reinterpret_cast<uintptr_t>(v.profile) & 15u) return fail(ctx, KVS_E_ARG, "eval_out: profile must be 16-byte aligned");
  if (!do_profile) v.profile = nullptr;
  if (P == 0) return KVS_OK;
  const int64_t N = inst->n_jobs_total, I = inst->n_instances, max_n = inst->max_jobs_per_instance;
  const Layout L = make_layout(N, I, max_n, rg ? rg->P_total : P, false);
  if (L.total > ctx->workspace_bytes)
    return fail(ctx, KVS_E_CAPACITY, "workspace too small for this call (see kvs_workspace_bytes)");
  cudaError_t ce = cudaSetDevice(ctx->device);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "cudaSetDevice");
  // everything the call uploads is laid out in one staging slot
  kvs_ctx::Stage* stg = nullptr;
  ce = take_stage(ctx, call_bytes(P), &stg);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "staging");
  unsigned long long* const init = reinterpret_cast<unsigned long long*>(stg->p);
  kvs_setting* const st_host = reinterpret_cast<kvs_setting*>(stg->p + CALL_COUNTERS);
  int64_t* const ids = reinterpret_cast<int64_t*>(st_host + P);       // full variant first, then the light one (P entries in all)
  int64_t* const after = ids + 2 * P;                                  // dynamic refill first, then speculative runs
  std::memset(init, 0, CALL_COUNTERS);
  const int parts = parts_for(P, max_n);
  if (parts > 1) std::memset(after + P, 0, static_cast<size_t>(P) * sizeof(FusedShare));
  std::memcpy(st_host, settings, static_cast<size_t>(P) * sizeof(kvs_setting));
  // Dynamic refill: the fused kernels form the batching schedule; a last kernel refills it in place.
  // Speculative runs: the same on top of the slicing schedule.
  int64_t n_refill = 0, n_spec = 0;
  for (int64_t e = 0; e < P; ++e)
    if (st_host[e].family == KVS_GBAD) { after[n_refill++] = e; st_host[e].family = KVS_GBA; }
  for (int64_t e = 0; e < P; ++e)
    if (st_host[e].family == KVS_GSAS) { after[n_refill + n_spec++] = e; st_host[e].family = KVS_GSA; }
  // one evaluation occupies its CTA from start to end, and small budgets take longest: those first
  auto by_budget = [&](int64_t x, int64_t y) { return st_host[x].M < st_host[y].M; };
  std::stable_sort(after, after + n_refill, by_budget);
  std::stable_sort(after + n_refill, after + n_refill + n_spec, by_budget);
  // The on-chip kernel of the speculative runs takes a few evaluations of one instance per CTA, smallest budgets first.
  int64_t* const groups = reinterpret_cast<int64_t*>(stg->p + groups_at(P));
  SpecShape shape;
  if (n_spec) {
    std::vector<int64_t> by_inst(after + n_refill, after + n_refill + n_spec);
    std::stable_sort(by_inst.begin(), by_inst.end(), [&](int64_t x, int64_t y) { return st_host[x].instance < st_host[y].instance; });
    std::vector<int64_t> evals_of;
    for (size_t i = 0; i < by_inst.size(); ++i) {
      if (i == 0 || st_host[by_inst[i]].instance != st_host[by_inst[i - 1]].instance) evals_of.push_back(0);
      ++evals_of.back();
    }
    shape = kvs_spec_shape(max_n, evals_of, ctx->sm_count);
    if (shape.warps > 0) {
      std::vector<std::pair<size_t, size_t>> cut;         // [first, last) of by_inst
      size_t at = 0;
      for (int64_t c : evals_of) {
        const int64_t pieces = spec_groups(c, shape.warps);
        for (int64_t g = 0; g < pieces; ++g) {
          const size_t size = static_cast<size_t>(c / pieces + (g < c % pieces ? 1 : 0));
          cut.emplace_back(at, at + size);
          at += size;
        }
      }
      std::stable_sort(cut.begin(), cut.end(), [&](const auto& x, const auto& y) { return st_host[by_inst[x.first]].M < st_host[by_inst[y.first]].M; });
      for (size_t g = 0; g < cut.size(); ++g)
        for (size_t i = 0; i < KVS_SPEC_GROUP; ++i)
          groups[KVS_SPEC_GROUP * g + i] = cut[g].first + i < cut[g].second ? by_inst[cut[g].first + i] : -1;
    }
  }
  if (n_refill || n_spec) {
    if (do_profile && (!o.job_start || !o.job_completion || !v.profile || o.job_start64 || o.job_completion64 || run_out))
      return fail(ctx, KVS_E_ARG, "the dynamic refill and speculative runs need job_start, job_completion and a profile (32-bit, no run list): they are their working storage");
    if (do_profile && (!v.horizon || !v.status))
      return fail(ctx, KVS_E_ARG, "the dynamic refill and speculative runs need the horizon and status outputs");
  }
  settings = st_host;

  unsigned char* ws = ctx->workspace;
  const int lane = rg ? rg->lane : -1;
  cudaStream_t const stream = lane >= 0 ? ctx->side[2 * lane + 1].stream : ctx->stream;
  const int64_t i0 = rg ? rg->i0 : 0, n_inst = rg ? rg->i1 - rg->i0 : I;
  unsigned char* const call = ws + L.call + (rg ? call_bytes(rg->e0) + static_cast<size_t>(rg->chunk) * CALL_COUNTERS : 0);
  ull* const counters = reinterpret_cast<ull*>(call);
  const kvs_setting* const settings_dev = reinterpret_cast<const kvs_setting*>(call + CALL_COUNTERS);
  FusedShare* const shares_dev = reinterpret_cast<FusedShare*>(call + lists_bytes(P));
  i64* const ids_dev = reinterpret_cast<i64*>(call + CALL_COUNTERS + static_cast<size_t>(P) * sizeof(kvs_setting));

  bool need_order = inst->o_est != nullptr;
  for (int64_t e = 0; e < P && !need_order; ++e) need_order = settings[e].family != KVS_GSA;

  SortParams sp{};
  // the ordering kernel numbers its instances from 0: a sub-range shifts the per-instance arrays
  sp.job_off = inst->job_off + i0; sp.s = inst->s; sp.o = inst->o; sp.key = inst->o_est; sp.arrival = inst->arrival;
  sp.window = inst->window; sp.n_instances = n_inst; sp.max_jobs = max_n; sp.need_order = need_order ? 1 : 0;
  sp.stats = reinterpret_cast<InstStats*>(ws + L.stats) + i0;
  sp.perm = reinterpret_cast<int32_t*>(ws + L.perm);
  sp.perm_tmp = reinterpret_cast<int32_t*>(ws + L.perm_tmp);
  sp.iperm = reinterpret_cast<int32_t*>(ws + L.iperm);
  sp.sorted_s = reinterpret_cast<int32_t*>(ws + L.sorted_s);
  sp.sorted_o = reinterpret_cast<int32_t*>(ws + L.sorted_o);
  sp.sorted_key = reinterpret_cast<int32_t*>(ws + L.sorted_key);
  // SPS / SimS evaluations that ask for no profile take the peak from run ends instead of rounds;
  // that needs prefix sums of s in key order (exact keys only)
  bool event_form = false;
  if (do_profile && !inst->o_est)
    for (int64_t e = 0; e < P && !event_form; ++e) event_form = settings[e].family >= KVS_SPS;
  sp.prefix_s = event_form ? reinterpret_cast<i64*>(ws + L.prefix_s) + i0 : nullptr;   // instance j writes at job_off[j] + j
  // The 32-bit fast kernel covers calls that want neither the explicit run list nor 64-bit job
  // results; evaluations it cannot finish (times of 2^31 or more, memory bound of 2^32 or more)
  // come back in a list that the general kernel works off.  Other calls go to the general kernel.
  const bool fast = !run_out && !o.job_start64 && !o.job_completion64;
  // Two variants of the fast kernel.  The light one (no ring, three CTAs per SM) takes the
  // evaluations that walk no rounds: all of them when no profile is formed, else the SPS / SimS
  // ones (and batching where none is stored), of which it passes on those that turn out to want their profile.  The full one takes
  // the geometric evaluations, listed here on the host, and what the light one passed on.
  // Without estimates every family has its own instantiation of the kernel and its own part of the
  // list: in the full variant the slicing algorithm first, then the batching one.  The kernels of a call run
  // one after the other, so a call that leaves most of the GPU idle anyway (at most one evaluation per SM) is not
  // split: one launch takes all its evaluations side by side.  (Evaluations of one family that are too large to be shared between
  // CTAs are side by side in their family's kernel too, which spills less: a call for one evaluation of a million jobs with its profile, in ms,
  // GBA 14.83 in the kernel for any family, 13.47 in its own, GSA 14.07 and 12.24.)
  bool one_family = true;
  for (int64_t e = 1; e < P && one_family; ++e) one_family = settings[e].family == settings[0].family;
  const bool one_wave = P <= ctx->sm_count && (parts > 1 || !one_family || inst->o_est);
  const bool split = inst->o_est == nullptr && !one_wave;
  int64_t n_full = 0, n_light = 0;
  int64_t full_of[4] = {0, 0, 0, 0}, light_of[4] = {0, 0, 0, 0};
  if (fast) {
    const bool all_full = one_wave && do_profile;
    // (the batching algorithm on exact keys takes its peak from run ends as well where no profile is stored; its variants with
    // a profile are the general kernel's, so the light variant sees them first)
    const bool gba_light = !inst->o_est && !v.profile;
    auto is_full = [&](int64_t e) {
      const kvs_setting& s = settings[e];
      return do_profile && (all_full || s.family == KVS_GSA || (s.family == KVS_GBA && !gba_light && !(split && (s.subroutine || s.per_class_s))));
    };
    // budgets below 2^31 and at most as many evaluations: order of the full list and number in one word
    const bool words = P < (1ll << 31);
    std::vector<uint64_t> order;
    if (words) order.reserve(static_cast<size_t>(P));
    for (int64_t e = 0; e < P; ++e) {
      if (!is_full(e)) { ids[P + n_light++] = e; continue; }
      ids[n_full++] = e;
      const uint64_t f = static_cast<uint64_t>(3 - settings[e].family), M = static_cast<uint64_t>(settings[e].M);
      if (words) order.push_back((split ? f << 62 | M << 31 : M << 33 | f << 31) | static_cast<uint64_t>(e));
    }
    // Longest first: the rounds of a schedule grow as the budget shrinks and the slicing algorithm
    // visits more runs than the batching one, and the CTAs draw evaluations in list order, so this
    // order keeps the last CTAs from finishing a long evaluation alone.
    if (words) {
      sort_above(order, 31);
      for (int64_t i = 0; i < n_full; ++i) ids[i] = static_cast<int64_t>(order[static_cast<size_t>(i)] & 0x7fffffffu);
    } else {
      std::stable_sort(ids, ids + n_full, [&](int64_t a, int64_t b) {
        if (split && settings[a].family != settings[b].family) return settings[a].family > settings[b].family;
        if (settings[a].M != settings[b].M) return settings[a].M < settings[b].M;
        return settings[a].family > settings[b].family;
      });
    }
    if (split) {
      if (!std::is_sorted(ids + P, ids + P + n_light, [&](int64_t a, int64_t b) { return settings[a].family < settings[b].family; }))
        std::stable_sort(ids + P, ids + P + n_light, [&](int64_t a, int64_t b) { return settings[a].family < settings[b].family; });
      for (int64_t i = 0; i < n_full; ++i) ++full_of[settings[ids[i]].family];
      for (int64_t i = 0; i < n_light; ++i) ++light_of[settings[ids[P + i]].family];
    }
    // [1] left-over count, [2] general work, [3] length of the full variant's list, [4] work of the full
    // variant for any family (starts behind the evaluations the family kernels take), [6] [7] work and
    // count of the light variant for any family, [8 + 2f] [9 + 2f] of the light kernel of family f,
    // [16 + 2f] [17 + 2f] of the full kernel of family f, [24] work of the speculative runs, [26] what their on-chip kernel leaves
    init[3] = static_cast<unsigned long long>(n_full);
    init[4] = static_cast<unsigned long long>(split ? n_full : 0);
    init[7] = static_cast<unsigned long long>(split ? 0 : n_light);
    for (int f = 0; f < 4; ++f) {
      init[9 + 2 * f] = static_cast<unsigned long long>(light_of[f]);
      init[17 + 2 * f] = static_cast<unsigned long long>(full_of[f]);
    }
  }
  const size_t upload = shape.groups ? call_bytes(P) : (parts > 1 ? groups_at(P) : lists_bytes(P));
  ce = send_stage(stg, counters, upload, rg ? ctx->copy_stream : ctx->stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "copy of the settings and evaluation lists");
  if (rg && (rc = rg->feed())) return rc;
  // calls that time their stages keep them one after the other
  const bool beside = fast && split && n_full && (lane >= 0 || (n_light && !ctx->timing));
  kvs_ctx::Side& side = ctx->side[lane >= 0 ? 2 * lane : 0];
  if (!beside && lane >= 0 && (ce = close_side(side, stream)) != cudaSuccess) return fail_cuda(ctx, ce, "stream ordering");

  if (ctx->timing && !rg) cudaEventRecord(ctx->ev[0], ctx->stream);
  ce = kvs_launch_sort(sp, ctx->sm_count * KVS_SORT_CTAS, stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "sort launch");
  if (ctx->timing && !rg) cudaEventRecord(ctx->ev[1], ctx->stream);

  BuildParams bp{};
  bp.job_off = inst->job_off; bp.s = inst->s; bp.o = inst->o; bp.key = inst->o_est; bp.arrival = inst->arrival;
  bp.window = inst->window; bp.n_instances = I; bp.max_jobs = max_n;
  bp.perm = sp.perm; bp.sorted_s = sp.sorted_s; bp.sorted_o = sp.sorted_o; bp.sorted_key = sp.sorted_key;
  bp.prefix_s = event_form ? reinterpret_cast<i64*>(ws + L.prefix_s) : nullptr;
  bp.iperm = sp.iperm;
  bp.stats = reinterpret_cast<InstStats*>(ws + L.stats);
  bp.settings = settings_dev;
  bp.fill = ctx->fill ? 1 : 0; bp.fill_job = ctx->fill_job; bp.fill_prof = ctx->fill_prof;
  bp.parts = 1;
  for (int64_t e = 0; e < P && !bp.variants; ++e) bp.variants = settings[e].subroutine || settings[e].per_class_s;
  bp.P = P; bp.out = o; bp.ev = v; bp.do_profile = do_profile;
  auto grid_for = [&](int ctas_per_sm, int64_t most) {
    int64_t g = static_cast<int64_t>(ctx->sm_count) * ctas_per_sm;
    if (g > most) g = most;
    return static_cast<int>(g);
  };
  // CTA scratch: a lane has its share of the grid that the workspace is sized for, else the call has all of it.  The kernels
  // beside start behind the light variant's.
  int64_t light_max = 0;
  for (int f = 0; f < 4; ++f) light_max = std::max(light_max, light_of[f]);
  const int64_t lane_ctas = lane >= 0 ? LANE_CTAS : KVS_MAX_GRID, lane_at = lane >= 0 ? lane * lane_ctas : 0;
  const int64_t light_ctas = !beside ? lane_ctas : (lane >= 0 ? rg->light_ctas : std::min(light_max, lane_ctas / 2)), side_at = lane_at + light_ctas;
  const int64_t side_ctas = beside ? lane_ctas - light_ctas : lane_ctas;
  auto scratch_at = [&](int64_t cta) {
    bp.lists = reinterpret_cast<int32_t*>(ws + L.lists + static_cast<size_t>(cta) * static_cast<size_t>(KVS_CTA_SCRATCH(max_n)));
    bp.fin_rank = reinterpret_cast<int32_t*>(ws + L.fin_rank) + cta * max_n;
  };
  scratch_at(lane_at);
  if (beside && (ce = open_side(side, stream, true)) != cudaSuccess) return fail_cuda(ctx, ce, "stream ordering");
  if (fast) {
    bp.slow_count = counters + 1;
    bp.slow_list = reinterpret_cast<i64*>(ws + L.slow_list) + (rg ? rg->e0 : 0);
    bp.walk_count = counters + 3;
    bp.walk_list = ids_dev;
    const i64* const light_list = ids_dev + P;
    auto launch_full = [&](cudaStream_t on) {
      int64_t at = 0;
      for (int f = KVS_GSA; f >= KVS_GBA; --f) {   // the order of the list
        if (full_of[f]) {
          bp.counter = counters + 16 + 2 * f;
          bp.eval_list = bp.walk_list + at;
          bp.eval_count = counters + 17 + 2 * f;
          const cudaError_t e = kvs_launch_fused(bp, grid_for(ctx->fused_ctas_per_sm, std::min(full_of[f], side_ctas)), 0, f, on);
          if (e != cudaSuccess) return e;
        }
        at += full_of[f];
      }
      return cudaSuccess;
    };
    if (beside) {
      scratch_at(side_at);
      if ((ce = launch_full(side.stream)) != cudaSuccess) return fail_cuda(ctx, ce, "fused launch");
      scratch_at(lane_at);
    }
    if (split) {
      int64_t at = 0;
      for (int f = 0; f < 4; ++f) {
        if (light_of[f]) {
          bp.counter = counters + 8 + 2 * f;
          bp.eval_list = light_list + at;
          bp.eval_count = counters + 9 + 2 * f;
          ce = kvs_launch_fused(bp, grid_for(ctx->light_ctas_per_sm, std::min(light_of[f], light_ctas)), 1, f, stream);
          if (ce != cudaSuccess) return fail_cuda(ctx, ce, "fused launch");
        }
        at += light_of[f];
      }
    } else if (n_light) {
      bp.counter = counters + 6;
      bp.eval_list = light_list;
      bp.eval_count = counters + 7;
      ce = kvs_launch_fused(bp, grid_for(ctx->light_ctas_per_sm, std::min(P, light_ctas)), 1, KVS_FUSED_ANY, stream);
      if (ce != cudaSuccess) return fail_cuda(ctx, ce, "fused launch");
    }
    if (ctx->timing && !rg) cudaEventRecord(ctx->ev[3], ctx->stream);
    if (split && !beside && (ce = launch_full(stream)) != cudaSuccess) return fail_cuda(ctx, ce, "fused launch");
    if (beside && lane < 0 && (ce = close_side(side, stream)) != cudaSuccess) return fail_cuda(ctx, ce, "stream ordering");
    // the light variant passes on what wants its rounds walked: nothing when no profile is formed, and nothing when
    // none is stored and the run ends give the peaks
    const bool passed_on = n_light && do_profile && (v.profile || inst->o_est);
    if (passed_on || (!split && n_full)) {
      // what the light variant passed on, and the evaluations of a call that is not split by family
      bp.counter = counters + 4;
      bp.eval_list = bp.walk_list;
      bp.eval_count = bp.walk_count;
      int grid = grid_for(ctx->fused_ctas_per_sm, std::min(P, lane_ctas));
      if (!split && n_full && !n_light) {
        bp.parts = parts;
        bp.shares = shares_dev;
        grid = static_cast<int>(std::min<int64_t>(P * bp.parts, static_cast<int64_t>(ctx->sm_count) * ctx->fused_ctas_per_sm));
      }
      ce = kvs_launch_fused(bp, grid, 0, bp.parts > 1 ? KVS_FUSED_SHARED : KVS_FUSED_ANY, stream);
      bp.parts = 1;
      if (ce != cudaSuccess) return fail_cuda(ctx, ce, "fused launch");
    }
    bp.eval_list = bp.slow_list;
    bp.eval_count = bp.slow_count;
  }
  bp.counter = counters + 2;
  int64_t most = std::min(P, lane_ctas);
  cudaStream_t last = stream;
  if (beside && lane >= 0) {
    // what the two variants leave to the general kernel: behind both
    if ((ce = open_side(side, stream, true)) != cudaSuccess) return fail_cuda(ctx, ce, "stream ordering");
    scratch_at(side_at);
    last = side.stream;
    most = std::min(P, side_ctas);
  }
  ce = kvs_launch_build(bp, grid_for(ctx->build_ctas_per_sm, most), last);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "build launch");
  if (do_profile && n_refill) {
    RefillParams rp{};
    rp.job_off = inst->job_off; rp.perm = sp.perm; rp.sorted_s = sp.sorted_s; rp.sorted_o = sp.sorted_o;
    rp.settings = settings_dev;
    rp.eval_list = ids_dev + 2 * P; rp.n_list = n_refill;
    rp.job_out_off = o.job_out_off; rp.job_start = o.job_start; rp.job_completion = o.job_completion;
    rp.profile_off = v.profile_off; rp.profile = v.profile;
    rp.peak = v.peak; rp.flow = v.flow; rp.horizon = v.horizon; rp.feasible = v.feasible; rp.status = v.status;
    ce = kvs_launch_refill(rp, ctx->stream);
    if (ce != cudaSuccess) return fail_cuda(ctx, ce, "refill launch");
  }
  if (do_profile && n_spec) {
    // the working storage is everything the ordering and fused kernels (and the refill) kept between them - the
    // orders, sorted copies, prefix sums and per-CTA scratch, one contiguous stretch of the workspace - free once
    // they have run
    SpecParams q{};
    q.job_off = inst->job_off; q.s = inst->s; q.o = inst->o;
    q.stats = reinterpret_cast<const InstStats*>(ws + L.stats);
    q.settings = settings_dev;
    q.eval_list = ids_dev + 2 * P + n_refill; q.n_list = n_spec;
    q.job_out_off = o.job_out_off; q.job_start = o.job_start; q.job_completion = o.job_completion;
    q.profile_off = v.profile_off; q.profile = v.profile;
    q.peak = v.peak; q.flow = v.flow; q.horizon = v.horizon; q.job_steps = v.job_steps; q.n_runs = o.n_runs;
    q.n_unfinished = v.n_unfinished; q.feasible = v.feasible; q.status = v.status;
    q.scratch = ws + L.perm; q.scratch_bytes = static_cast<i64>(L.slow_list - L.perm); q.max_jobs = max_n;
    const i64 room = static_cast<i64>(L.slow_list - L.perm) / kvs_spec_warp_bytes(max_n);
    const i64 want = static_cast<i64>(ctx->sm_count) * 32;
    q.n_warps = std::min<i64>(std::min<i64>(room, want), q.n_list);
    q.counter = counters + 24;
    // (its lists of participants take less of the working storage than the CTA scratch of as many evaluations; otherwise the other kernel takes them all)
    q.groups = reinterpret_cast<const i64*>(call + groups_at(P)); q.n_groups = shape.groups * spec_list_bytes(max_n, shape.warps) <= q.scratch_bytes ? shape.groups : 0;
    q.group_warps = shape.warps; q.ring = shape.ring;
    q.left_list = reinterpret_cast<i64*>(ws + L.slow_list); q.left_count = counters + 26;   // the general kernel has run: its list is free
    ce = kvs_launch_spec(q, ctx->stream);
    if (ce != cudaSuccess) return fail_cuda(ctx, ce, "launch of the speculative runs");
  }
  if (ctx->timing && !rg) { cudaEventRecord(ctx->ev[2], ctx->stream); ctx->timed = true; ctx->split_timed = fast; }
  return KVS_OK;
}

// A device entry point.  Where it fails half-way, what it has launched on a stream of its own is put in front of whatever the
// caller does next on the context's stream.
int run_fused(kvs_ctx* ctx, const kvs_instances* inst, const kvs_setting* settings, int64_t P,
              const kvs_schedule_out* out, const kvs_eval_out* ev, int do_profile) {
  if (!ctx) return KVS_E_STATE;
  const int rc = guarded(ctx, [&] { return enqueue_fused(ctx, inst, settings, P, out, ev, do_profile, nullptr); });
  if (rc) close_sides(ctx);
  return rc;
}

}  // namespace

extern "C" {

int kvs_init(const kvs_init_params* params, kvs_ctx** out) {
  if (!params || !out) return KVS_E_ARG;
  *out = nullptr;
  int count = 0;
  if (cudaGetDeviceCount(&count) != cudaSuccess || count <= 0) return KVS_E_CUDA;  // no CPU fallback exists
  if (params->device < 0 || params->device >= count) return KVS_E_ARG;
  if (params->workspace_bytes > 0 && !params->workspace) return KVS_E_ARG;
  if (reinterpret_cast<uintptr_t>(params->workspace) & 255u) return KVS_E_ARG;
  kvs_ctx* ctx = new (std::nothrow) kvs_ctx();
  if (!ctx) return KVS_E_STATE;
  ctx->device = params->device;
  ctx->stream = static_cast<cudaStream_t>(params->stream);
  ctx->workspace = static_cast<unsigned char*>(params->workspace);
  ctx->workspace_bytes = params->workspace_bytes;
  cudaDeviceProp prop;
  if (cudaSetDevice(ctx->device) != cudaSuccess || cudaGetDeviceProperties(&prop, ctx->device) != cudaSuccess) {
    delete ctx;
    return KVS_E_CUDA;
  }
  ctx->sm_count = prop.multiProcessorCount;
  ctx->build_ctas_per_sm = kvs_build_ctas_per_sm();
  ctx->fused_ctas_per_sm = kvs_fused_ctas_per_sm(0);
  ctx->light_ctas_per_sm = kvs_fused_ctas_per_sm(1);
  if (kvs_setup_sort() != cudaSuccess || kvs_setup_generic() != cudaSuccess || kvs_setup_bounds() != cudaSuccess || kvs_setup_spec() != cudaSuccess) {
    delete ctx;
    return KVS_E_CUDA;
  }
  *out = ctx;
  return KVS_OK;
}

int kvs_destroy(kvs_ctx* ctx) {
  if (ctx) {
    for (cudaEvent_t e : ctx->ev) if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : ctx->chunk_ev) if (e) cudaEventDestroy(e);
    if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
    for (kvs_ctx::Side& s : ctx->side) {
      if (s.from) cudaEventDestroy(s.from);
      if (s.done) cudaEventDestroy(s.done);
      if (s.stream) cudaStreamDestroy(s.stream);
    }
    if (ctx->pinned) cudaFreeHost(ctx->pinned);
    for (kvs_ctx::Stage& s : ctx->stage) {
      if (s.used) cudaEventSynchronize(s.done);
      if (s.done) cudaEventDestroy(s.done);
      if (s.p) cudaFreeHost(s.p);
    }
  }
  delete ctx;
  return KVS_OK;
}

int kvs_set_unwritten(kvs_ctx* ctx, int32_t enabled, int32_t job_value, int32_t profile_value) {
  if (!ctx) return KVS_E_STATE;
  ctx->fill = enabled != 0;
  ctx->fill_job = job_value;
  ctx->fill_prof = profile_value;
  return KVS_OK;
}

int kvs_reader_open(int32_t device, kvs_reader** out) {
  if (!out) return KVS_E_ARG;
  *out = nullptr;
  int count = 0;
  if (cudaGetDeviceCount(&count) != cudaSuccess || count <= 0) return KVS_E_CUDA;
  if (device < 0 || device >= count) return KVS_E_ARG;
  kvs_reader* r = new (std::nothrow) kvs_reader();
  if (!r) return KVS_E_STATE;
  r->device = device;
  if (cudaSetDevice(device) != cudaSuccess || cudaEventCreateWithFlags(&r->sent, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&r->arrived, cudaEventDisableTiming) != cudaSuccess) {
    kvs_reader_close(r);
    return KVS_E_CUDA;
  }
  *out = r;
  return KVS_OK;
}

int kvs_reader_close(kvs_reader* r) {
  if (r) {
    if (r->open) cudaEventSynchronize(r->arrived);         // begun and never ended
    if (r->sending) cudaEventSynchronize(r->sent);
    for (cudaEvent_t e : {r->arrived, r->sent}) if (e) cudaEventDestroy(e);
    for (kvs_reader::Pinned* m : {&r->in, &r->rows}) if (m->p) cudaFreeHost(m->p);
  }
  delete r;
  return KVS_OK;
}

const char* kvs_reader_error(const kvs_reader* r) { return r ? r->err.c_str() : "no reader"; }

// Room for at least `bytes` bytes in memory that nothing in flight uses.
static cudaError_t make_room(kvs_reader::Pinned& m, size_t bytes) {
  if (m.bytes >= bytes) return cudaSuccess;
  if (m.p) cudaFreeHost(m.p);
  m.p = nullptr; m.bytes = 0;
  const size_t want = bytes + bytes / 2 + 4096;
  const cudaError_t ce = cudaMallocHost(reinterpret_cast<void**>(&m.p), want);
  if (ce == cudaSuccess) m.bytes = want;
  return ce;
}

int kvs_sizes_begin(kvs_reader* r, void* stream, const int64_t* job_off, int64_t n_instances, const int64_t* capacity, int64_t P) {
  if (!r) return KVS_E_STATE;
  if (r->open) return fail(r, KVS_E_STATE, "sizes: this reader's last request has not been ended");
  if (n_instances < 0 || P < 0) return fail(r, KVS_E_ARG, "sizes: negative count");
  r->stream = static_cast<cudaStream_t>(stream);
  r->n_off = job_off ? n_instances + 1 : -1;
  r->n_cap = capacity ? P : -1;
  const size_t off_bytes = job_off ? static_cast<size_t>(n_instances + 1) * 8 : 0, cap_bytes = capacity ? static_cast<size_t>(P) * 8 : 0;
  cudaError_t ce = cudaSetDevice(r->device);
  if (ce == cudaSuccess) ce = make_room(r->in, off_bytes + cap_bytes);
  if (ce == cudaSuccess && off_bytes) ce = cudaMemcpyAsync(r->in.p, job_off, off_bytes, cudaMemcpyDeviceToHost, r->stream);
  const bool under_way = ce == cudaSuccess;
  if (ce == cudaSuccess && cap_bytes) ce = cudaMemcpyAsync(reinterpret_cast<unsigned char*>(r->in.p) + off_bytes, capacity, cap_bytes, cudaMemcpyDeviceToHost, r->stream);
  if (ce == cudaSuccess) ce = cudaEventRecord(r->arrived, r->stream);
  if (ce != cudaSuccess) {
    if (under_way) cudaStreamSynchronize(r->stream);
    return fail_cuda(r, ce, "read of the sizes");
  }
  r->open = true;
  return KVS_OK;
}

static int sizes_end(kvs_reader* r, const kvs_setting* settings, int64_t P, int64_t* job_out_off, int64_t* profile_off, kvs_sizes* out) {
  if (!r->open) return fail(r, KVS_E_STATE, "sizes: not begun");
  r->open = false;
  cudaError_t ce = cudaSetDevice(r->device);
  const cudaError_t waited = cudaEventSynchronize(r->arrived);
  if (ce == cudaSuccess) ce = waited;
  if (ce != cudaSuccess) return fail_cuda(r, ce, "read of the sizes");
  if (P < 0 || (job_out_off && (r->n_off < 1 || (P > 0 && !settings))) || (profile_off && r->n_cap != P)) return fail(r, KVS_E_ARG, "sizes: not those that were asked for");
  const int64_t *off = r->in.p, *cap = r->in.p + (r->n_off > 0 ? r->n_off : 0);
  kvs_sizes s{};
  for (int64_t i = 0; i + 1 < r->n_off; ++i) s.max_jobs = std::max(s.max_jobs, off[i + 1] - off[i]);
  if (job_out_off)
    for (int64_t e = 0; e < P; ++e)
      if (settings[e].instance < 0 || settings[e].instance + 1 >= r->n_off) return fail(r, KVS_E_ARG, "settings: instance out of range");
  // a negative count would move the offsets behind it in front of what is reserved for them
  for (int64_t e = 0; e < r->n_cap; ++e)
    if (cap[e] < 0) return fail(r, KVS_E_ARG, "sizes: negative capacity");
  if (job_out_off || profile_off) {
    const size_t row = static_cast<size_t>(P) + 1;
    if (r->sending && (ce = cudaEventSynchronize(r->sent)) != cudaSuccess) return fail_cuda(r, ce, "copy of the offsets");
    r->sending = false;
    if ((ce = make_room(r->rows, 16 * row)) != cudaSuccess) return fail_cuda(r, ce, "cudaMallocHost");
    int64_t* const rows = r->rows.p;
    auto fill = [&](int64_t* at, auto count) {
      int64_t sum = 0;
      for (int64_t e = 0; e < P; ++e) { at[e] = sum; sum += count(e); }
      return at[P] = sum;
    };
    if (job_out_off) s.job_results = fill(rows, [&](int64_t e) { return std::max<int64_t>(0, off[settings[e].instance + 1] - off[settings[e].instance]); });
    if (profile_off) s.profile_rounds = fill(rows + row, [&](int64_t e) { return cap[e]; });
    if (job_out_off && profile_off == job_out_off + row) {               // one piece
      ce = cudaMemcpyAsync(job_out_off, rows, 16 * row, cudaMemcpyHostToDevice, r->stream);
    } else {
      if (job_out_off) ce = cudaMemcpyAsync(job_out_off, rows, 8 * row, cudaMemcpyHostToDevice, r->stream);
      if (ce == cudaSuccess && profile_off) ce = cudaMemcpyAsync(profile_off, rows + row, 8 * row, cudaMemcpyHostToDevice, r->stream);
    }
    const cudaError_t marked = cudaEventRecord(r->sent, r->stream);
    r->sending = marked == cudaSuccess;
    if (!r->sending) cudaStreamSynchronize(r->stream);                   // no event to wait for later
    if (ce == cudaSuccess) ce = marked;
    if (ce != cudaSuccess) return fail_cuda(r, ce, "copy of the offsets");
  }
  if (out) *out = s;
  return KVS_OK;
}
int kvs_sizes_end(kvs_reader* r, const kvs_setting* settings, int64_t P, int64_t* job_out_off, int64_t* profile_off, kvs_sizes* out) {
  if (!r) return KVS_E_STATE;
  return guarded(r, [&] { return sizes_end(r, settings, P, job_out_off, profile_off, out); });
}

const char* kvs_last_error(const kvs_ctx* ctx) { return ctx ? ctx->err.c_str() : "no context"; }

int kvs_set_timing(kvs_ctx* ctx, int32_t enabled) {
  if (!ctx) return KVS_E_STATE;
  if (enabled && !ctx->ev[0]) {
    if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(ctx, KVS_E_CUDA, "cudaSetDevice");
    for (cudaEvent_t& e : ctx->ev)
      if (cudaEventCreate(&e) != cudaSuccess) return fail(ctx, KVS_E_CUDA, "cudaEventCreate");
  }
  ctx->timing = enabled != 0;
  ctx->timed = false;
  return KVS_OK;
}

int kvs_last_timing(kvs_ctx* ctx, float* sort_ms, float* build_ms) {
  if (!ctx) return KVS_E_STATE;
  if (sort_ms) *sort_ms = 0.f;
  if (build_ms) *build_ms = 0.f;
  if (!ctx->timed) return KVS_OK;
  cudaError_t ce = cudaEventSynchronize(ctx->ev[2]);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "cudaEventSynchronize");
  if (sort_ms) cudaEventElapsedTime(sort_ms, ctx->ev[0], ctx->ev[1]);
  if (build_ms) cudaEventElapsedTime(build_ms, ctx->ev[1], ctx->ev[2]);
  return KVS_OK;
}

int kvs_last_timing_split(kvs_ctx* ctx, float* sort_ms, float* light_ms, float* full_ms) {
  if (!ctx) return KVS_E_STATE;
  if (sort_ms) *sort_ms = 0.f;
  if (light_ms) *light_ms = 0.f;
  if (full_ms) *full_ms = 0.f;
  if (!ctx->timed) return KVS_OK;
  cudaError_t ce = cudaEventSynchronize(ctx->ev[2]);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "cudaEventSynchronize");
  if (sort_ms) cudaEventElapsedTime(sort_ms, ctx->ev[0], ctx->ev[1]);
  // the event between the two variants exists only on the fast path
  if (cudaEventQuery(ctx->ev[3]) == cudaSuccess && ctx->split_timed) {
    if (light_ms) cudaEventElapsedTime(light_ms, ctx->ev[1], ctx->ev[3]);
    if (full_ms) cudaEventElapsedTime(full_ms, ctx->ev[3], ctx->ev[2]);
  } else if (full_ms) {
    cudaEventElapsedTime(full_ms, ctx->ev[1], ctx->ev[2]);
  }
  return KVS_OK;
}

int kvs_debug_check_word(uint64_t* word, int32_t* compiled_in, int32_t reset) {
  unsigned long long w = 0ull;
  int compiled = 0;
  if (cudaDeviceSynchronize() != cudaSuccess) return KVS_E_CUDA;
  if (kvs_fused_check_word(&w, &compiled, reset) != cudaSuccess) return KVS_E_CUDA;
  // the kernels of the sequential rules keep words of their own: the first violation found is reported
  unsigned long long w2 = 0ull, w3 = 0ull;
  if (kvs_refill_check_word(&w2, nullptr, reset) != cudaSuccess || kvs_spec_check_word(&w3, nullptr, reset) != cudaSuccess)
    return KVS_E_CUDA;
  if (w == 0ull) w = w2 ? w2 : w3;
  if (word) *word = w;
  if (compiled_in) *compiled_in = compiled;
  return KVS_OK;
}

int kvs_workspace_bytes(int64_t n_jobs_total, int64_t n_instances, int64_t max_jobs_per_instance,
                        int64_t n_evaluations, int64_t generic_capacity, int32_t host_staging, uint64_t* out) {
  if (!out || n_jobs_total < 0 || n_instances < 0 || max_jobs_per_instance < 0 || n_evaluations < 0 || generic_capacity < 0)
    return KVS_E_ARG;
  size_t need = make_layout(n_jobs_total, n_instances, max_jobs_per_instance, n_evaluations, host_staging != 0).total;
  if (generic_capacity > 0) {
    const size_t g = make_generic_layout(generic_capacity, n_evaluations).total;
    if (g > need) need = g;
  }
  const size_t w = make_sweep_layout(max_jobs_per_instance).total;
  if (w > need) need = w;
  *out = need;
  return KVS_OK;
}

int kvs_build_schedule(kvs_ctx* ctx, const kvs_instances* inst, const kvs_setting* settings, int64_t P,
                       const kvs_schedule_out* out, const kvs_eval_out* ev) {
  return run_fused(ctx, inst, settings, P, out, ev, 0);
}

int kvs_evaluate_built(kvs_ctx* ctx, const kvs_instances* inst, const kvs_setting* settings, int64_t P,
                       const kvs_schedule_out* out, const kvs_eval_out* ev) {
  return run_fused(ctx, inst, settings, P, out, ev, 1);
}

static int evaluate_built_host(kvs_ctx* ctx, const kvs_instances* inst, const kvs_setting* settings, int64_t P, const kvs_eval_out* ev, bool* begun) {
  int rc = check_instances(ctx, inst);
  if (rc) return rc;
  if (!ev) return fail(ctx, KVS_E_ARG, "eval_out: null");
  if (ev->profile) return fail(ctx, KVS_E_ARG, "host entry point returns scalars only (profile must be NULL)");
  rc = check_settings(ctx, inst, settings, P);
  if (rc) return rc;
  for (int64_t e = 0; e < P; ++e)
    if (settings[e].family == KVS_GBAD || settings[e].family == KVS_GSAS)
      return fail(ctx, KVS_E_ARG, "the host entry point takes neither the dynamic refill nor speculative runs (they need per-job results and a profile on the device)");
  const int64_t N = inst->n_jobs_total, I = inst->n_instances;
  for (int64_t i = 0; i < I; ++i)
    if (inst->job_off[i] < 0 || inst->job_off[i + 1] < inst->job_off[i] || inst->job_off[i + 1] > N)
      return fail(ctx, KVS_E_ARG, "instances: job_off is not nondecreasing within [0, n_jobs_total]");
  const Layout L = make_layout(N, I, inst->max_jobs_per_instance, P, true);
  if (L.total > ctx->workspace_bytes) return fail(ctx, KVS_E_CAPACITY, "workspace too small for host staging (see kvs_workspace_bytes)");
  cudaError_t ce = cudaSetDevice(ctx->device);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "cudaSetDevice");
  if (!ctx->copy_stream && (ce = cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking)) != cudaSuccess)
    return fail_cuda(ctx, ce, "cudaStreamCreate");
  for (cudaEvent_t& e : ctx->chunk_ev)
    if (!e && (ce = cudaEventCreateWithFlags(&e, cudaEventDisableTiming)) != cudaSuccess) return fail_cuda(ctx, ce, "cudaEventCreate");
  unsigned char* ws = ctx->workspace;

  // Evaluations are worked off chunk of instances by chunk of instances, so that the copy of the
  // next chunk's jobs overlaps the kernels of the current one: order them by instance (stable).
  std::vector<int64_t> order(static_cast<size_t>(P));
  for (int64_t e = 0; e < P; ++e) order[static_cast<size_t>(e)] = e;
  bool identity = true;
  for (int64_t e = 1; e < P && identity; ++e) identity = settings[e - 1].instance <= settings[e].instance;
  if (!identity)
    std::stable_sort(order.begin(), order.end(), [&](int64_t a, int64_t b) { return settings[a].instance < settings[b].instance; });
  std::vector<kvs_setting> sorted(static_cast<size_t>(P));
  for (int64_t r = 0; r < P; ++r) sorted[static_cast<size_t>(r)] = settings[order[static_cast<size_t>(r)]];

  kvs_instances dev = *inst;
  dev.job_off = reinterpret_cast<const int64_t*>(ws + L.st_off);
  dev.s = reinterpret_cast<const int32_t*>(ws + L.st_s);
  dev.o = reinterpret_cast<const int32_t*>(ws + L.st_o);
  dev.o_est = inst->o_est ? reinterpret_cast<const int32_t*>(ws + L.st_key) : nullptr;
  dev.arrival = inst->arrival ? reinterpret_cast<const int64_t*>(ws + L.st_arr) : nullptr;
  kvs_eval_out d{};
  d.peak = reinterpret_cast<int64_t*>(ws + L.sc_peak);
  d.flow = reinterpret_cast<int64_t*>(ws + L.sc_flow);
  d.job_steps = reinterpret_cast<int64_t*>(ws + L.sc_steps);
  d.horizon = reinterpret_cast<int64_t*>(ws + L.sc_hor);
  d.n_unfinished = reinterpret_cast<int64_t*>(ws + L.sc_unf);
  d.feasible = reinterpret_cast<uint8_t*>(ws + L.sc_feas);
  d.status = reinterpret_cast<int32_t*>(ws + L.sc_stat);

  *begun = true;
  // the staging areas may still be read by earlier work on the context's stream
  if ((ce = cudaEventRecord(ctx->chunk_ev[KVS_HOST_CHUNKS], ctx->stream)) != cudaSuccess ||
      (ce = cudaStreamWaitEvent(ctx->copy_stream, ctx->chunk_ev[KVS_HOST_CHUNKS], 0)) != cudaSuccess)
    return fail_cuda(ctx, ce, "stream ordering");
  ce = cudaMemcpyAsync(ws + L.st_off, inst->job_off, static_cast<size_t>(I + 1) * 8, cudaMemcpyHostToDevice, ctx->copy_stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "host-to-device copy of job_off");
  // Chunks of about KVS_CHUNK_EVALS evaluations, at most KVS_HOST_CHUNKS of them: large enough that their launches do not
  // count (256: 4.7 ms in the example above), small enough that the last one, whose kernels run behind the last copy, is a
  // small part of the work (1,024: 3.95 ms).  The lanes share the CTA scratch, which smaller calls have less of.
  int64_t n_chunks = P < KVS_MAX_GRID ? 1 : P / KVS_CHUNK_EVALS;
  if (n_chunks > KVS_HOST_CHUNKS) n_chunks = KVS_HOST_CHUNKS;
  if (n_chunks > I) n_chunks = I;
  if (n_chunks < 1) n_chunks = 1;
  for (int l = 0; l < KVS_LANES && n_chunks > 1; ++l)
    if ((ce = open_side(ctx->side[2 * l + 1], ctx->stream, false)) != cudaSuccess) return fail_cuda(ctx, ce, "stream ordering");
  const int64_t light_ctas = lane_light_ctas(settings, P);
  int64_t r0 = 0;
  for (int64_t c = 0; c < n_chunks; ++c) {
    const int64_t i0 = c * I / n_chunks, i1 = (c + 1) * I / n_chunks;
    const int lane = n_chunks > 1 ? static_cast<int>(c % KVS_LANES) : -1;
    const int64_t j0 = I ? inst->job_off[i0] : 0, j1 = I ? inst->job_off[i1] : 0;
    const size_t cnt = static_cast<size_t>(j1 - j0);
    auto h2d = [&](size_t off, const void* src, size_t elem) {
      return (src && cnt) ? cudaMemcpyAsync(ws + off + static_cast<size_t>(j0) * elem, static_cast<const unsigned char*>(src) + static_cast<size_t>(j0) * elem,
                                            cnt * elem, cudaMemcpyHostToDevice, ctx->copy_stream)
                          : cudaSuccess;
    };
    auto feed = [&]() -> int {
      if ((ce = h2d(L.st_s, inst->s, 4)) != cudaSuccess || (ce = h2d(L.st_o, inst->o, 4)) != cudaSuccess ||
          (ce = h2d(L.st_key, inst->o_est, 4)) != cudaSuccess || (ce = h2d(L.st_arr, inst->arrival, 8)) != cudaSuccess)
        return fail_cuda(ctx, ce, "host-to-device copy of the instances");
      if ((ce = cudaEventRecord(ctx->chunk_ev[c], ctx->copy_stream)) != cudaSuccess ||
          (ce = cudaStreamWaitEvent(lane >= 0 ? ctx->side[2 * lane + 1].stream : ctx->stream, ctx->chunk_ev[c], 0)) != cudaSuccess)
        return fail_cuda(ctx, ce, "stream ordering");
      return KVS_OK;
    };
    int64_t r1 = r0;
    while (r1 < P && sorted[static_cast<size_t>(r1)].instance < i1) ++r1;
    if (r1 > r0) {
      kvs_eval_out dc = d;
      dc.peak += r0; dc.flow += r0; dc.job_steps += r0; dc.horizon += r0; dc.n_unfinished += r0; dc.feasible += r0; dc.status += r0;
      const FusedRange rg{i0, i1, r0, P, static_cast<int>(c), lane, light_ctas, feed};
      rc = enqueue_fused(ctx, &dev, sorted.data() + r0, r1 - r0, nullptr, &dc, 1, &rg);
      if (rc) return rc;
    } else if ((rc = feed()) != KVS_OK) {
      return rc;
    }
    r0 = r1;
  }

  if ((ce = close_sides(ctx)) != cudaSuccess) return fail_cuda(ctx, ce, "stream ordering");

  // results come back in the order the evaluations were worked off
  const size_t p8 = static_cast<size_t>(P) * 8;
  std::vector<int64_t> t64;
  std::vector<int32_t> t32;
  std::vector<uint8_t> t8;
  auto fetch = [&](void* dst, size_t off, size_t elem) -> cudaError_t {
    if (!dst || P == 0) return cudaSuccess;
    if (identity) return cudaMemcpyAsync(dst, ws + off, static_cast<size_t>(P) * elem, cudaMemcpyDeviceToHost, ctx->stream);
    // scattered back through a temporary once the stream has finished
    return cudaSuccess;
  };
  if ((ce = fetch(ev->peak, L.sc_peak, 8)) != cudaSuccess || (ce = fetch(ev->flow, L.sc_flow, 8)) != cudaSuccess ||
      (ce = fetch(ev->job_steps, L.sc_steps, 8)) != cudaSuccess || (ce = fetch(ev->horizon, L.sc_hor, 8)) != cudaSuccess ||
      (ce = fetch(ev->n_unfinished, L.sc_unf, 8)) != cudaSuccess || (ce = fetch(ev->feasible, L.sc_feas, 1)) != cudaSuccess ||
      (ce = fetch(ev->status, L.sc_stat, 4)) != cudaSuccess)
    return fail_cuda(ctx, ce, "device-to-host copy of the results");
  ce = cudaStreamSynchronize(ctx->stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "stream synchronize");
  if (!identity && P > 0) {
    t64.resize(static_cast<size_t>(P)); t32.resize(static_cast<size_t>(P)); t8.resize(static_cast<size_t>(P));
    auto back64 = [&](int64_t* dst, size_t off) -> cudaError_t {
      if (!dst) return cudaSuccess;
      const cudaError_t e = cudaMemcpy(t64.data(), ws + off, p8, cudaMemcpyDeviceToHost);
      if (e == cudaSuccess) for (int64_t r = 0; r < P; ++r) dst[order[static_cast<size_t>(r)]] = t64[static_cast<size_t>(r)];
      return e;
    };
    if ((ce = back64(ev->peak, L.sc_peak)) != cudaSuccess || (ce = back64(ev->flow, L.sc_flow)) != cudaSuccess ||
        (ce = back64(ev->job_steps, L.sc_steps)) != cudaSuccess || (ce = back64(ev->horizon, L.sc_hor)) != cudaSuccess ||
        (ce = back64(ev->n_unfinished, L.sc_unf)) != cudaSuccess)
      return fail_cuda(ctx, ce, "device-to-host copy of the results");
    if (ev->feasible) {
      if ((ce = cudaMemcpy(t8.data(), ws + L.sc_feas, static_cast<size_t>(P), cudaMemcpyDeviceToHost)) != cudaSuccess) return fail_cuda(ctx, ce, "device-to-host copy of the results");
      for (int64_t r = 0; r < P; ++r) ev->feasible[order[static_cast<size_t>(r)]] = t8[static_cast<size_t>(r)];
    }
    if (ev->status) {
      if ((ce = cudaMemcpy(t32.data(), ws + L.sc_stat, static_cast<size_t>(P) * 4, cudaMemcpyDeviceToHost)) != cudaSuccess) return fail_cuda(ctx, ce, "device-to-host copy of the results");
      for (int64_t r = 0; r < P; ++r) ev->status[order[static_cast<size_t>(r)]] = t32[static_cast<size_t>(r)];
    }
  }
  return KVS_OK;
}

int kvs_evaluate_built_host(kvs_ctx* ctx, const kvs_instances* inst, const kvs_setting* settings, int64_t P,
                            const kvs_eval_out* ev) {
  if (!ctx) return KVS_E_STATE;
  bool begun = false;                        // something may have been enqueued
  const int rc = guarded(ctx, [&] { return evaluate_built_host(ctx, inst, settings, P, ev, &begun); });
  if (rc && begun) {
    // Whatever has been enqueued before the failure is over before the caller, who may free or reuse the buffers, has the
    // status: the lanes and their side streams, the copies, then the context's stream.
    for (kvs_ctx::Side& sd : ctx->side)
      if (sd.open) { cudaStreamSynchronize(sd.stream); sd.open = false; }
    if (ctx->copy_stream) cudaStreamSynchronize(ctx->copy_stream);
    cudaStreamSynchronize(ctx->stream);
  }
  return rc;
}

static int check_runs(kvs_ctx* ctx, const kvs_runs* runs, const kvs_eval_out* ev) {
  if (!ctx) return KVS_E_STATE;
  if (!runs || !ev) return fail(ctx, KVS_E_ARG, "runs or eval_out is null");
  if (runs->P < 0) return fail(ctx, KVS_E_ARG, "runs: negative count");
  if (runs->P == 0) return KVS_OK;
  if (!runs->run_off || !runs->run_start || !runs->run_len || !runs->run_s) return fail(ctx, KVS_E_ARG, "runs: null array");
  if (!ev->profile_off) return fail(ctx, KVS_E_ARG, "eval_out: profile_off (capacities) is required");
  return KVS_OK;
}

int kvs_evaluate_schedule_sized(kvs_ctx* ctx, const kvs_runs* runs, const kvs_eval_out* ev, int64_t cap_total) {
  const int rc = check_runs(ctx, runs, ev);
  if (rc || runs->P == 0) return rc;
  if (cap_total < 0) return fail(ctx, KVS_E_ARG, "eval_out: negative capacity");
  cudaError_t ce = cudaSetDevice(ctx->device);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "cudaSetDevice");
  const GenericLayout L = make_generic_layout(cap_total, runs->P);
  if (L.total > ctx->workspace_bytes) return fail(ctx, KVS_E_CAPACITY, "workspace too small for the generic evaluator");
  unsigned char* ws = ctx->workspace;
  GenericParams gp{};
  gp.runs = *runs; gp.ev = *ev;
  gp.dconst = reinterpret_cast<i64*>(ws + L.dconst);
  gp.dcount = reinterpret_cast<int32_t*>(ws + L.dcount);
  gp.slots = cap_total + runs->P;
  gp.tile_peak = reinterpret_cast<u32*>(ws + L.peak);
  gp.tile_done = reinterpret_cast<u32*>(ws + L.done);
  gp.wide_list = reinterpret_cast<i64*>(ws + L.list);
  gp.wide_count = reinterpret_cast<u32*>(ws + L.count);
  gp.odd = gp.wide_count + 1;
  gp.fill = ctx->fill ? 1 : 0; gp.fill_prof = ctx->fill_prof;
  ce = cudaMemsetAsync(ws + L.count, 0, 8, ctx->stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "memset");
  ce = kvs_launch_generic_tiled(gp, cap_total, ctx->sm_count, ctx->stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "generic launch");
  return KVS_OK;
}

int kvs_evaluate_schedule(kvs_ctx* ctx, const kvs_runs* runs, const kvs_eval_out* ev) {
  const int rc = check_runs(ctx, runs, ev);
  if (rc || runs->P == 0) return rc;
  cudaError_t ce = cudaSetDevice(ctx->device);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "cudaSetDevice");
  // total capacity = profile_off[P]: one small synchronous read sizes the scratch arrays
  int64_t cap_total = 0;
  ce = cudaMemcpyAsync(&cap_total, ev->profile_off + runs->P, 8, cudaMemcpyDeviceToHost, ctx->stream);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(ctx->stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "read of profile_off");
  return kvs_evaluate_schedule_sized(ctx, runs, ev, cap_total);
}

int kvs_bounds(kvs_ctx* ctx, const kvs_instances* inst, const kvs_setting* settings, int64_t P, const kvs_bounds_out* out) {
  if (!ctx) return KVS_E_STATE;
  int rc = check_instances(ctx, inst);
  if (rc) return rc;
  if (!out) return fail(ctx, KVS_E_ARG, "bounds: out is null");
  if (inst->window != 0) return fail(ctx, KVS_E_ARG, "bounds: needs offline instances (window = 0)");
  if (P < 0 || (P > 0 && !settings)) return check_settings(ctx, inst, settings, P);
  if (P == 0) return KVS_OK;
  const int64_t I = inst->n_instances, max_n = inst->max_jobs_per_instance;
  const Layout L = make_layout(0, I, 0, P, false);           // settings and statistics only
  if (L.total > ctx->workspace_bytes) return fail(ctx, KVS_E_CAPACITY, "workspace too small for this call (see kvs_workspace_bytes)");
  cudaError_t ce = cudaSetDevice(ctx->device);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "cudaSetDevice");
  unsigned char* ws = ctx->workspace;
  kvs_ctx::Stage* stg = nullptr;
  ce = take_stage(ctx, static_cast<size_t>(P) * (sizeof(kvs_setting) + 16), &stg);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "staging");
  // The kernels read the settings straight from the page-locked slot, without an upload before them.  Where they differ only in
  // instance and budget, those two are all that goes there: eight bytes instead of 64, which is what a call of thousands of
  // settings spends its time on, on the host and on the link (8,192 settings: 98 us a call, 144 with all of them in full).
  kvs_setting* const geo = reinterpret_cast<kvs_setting*>(stg->p);
  int64_t* const runs = reinterpret_cast<int64_t*>(geo + P);
  int2* const brief = reinterpret_cast<int2*>(geo + 1);      // in place of the settings but the first
  // runs of evaluations of one instance, short enough that the runs of few instances still give every SM its three CTAs
  const int64_t longest = std::max<int64_t>(1, P / (3 * ctx->sm_count));
  int64_t n_runs = 0, length = 0;
  bool in_brief = P > 1 && I < (1ll << 31);
  // the family is not used: the settings are checked as geometric ones
  auto as_geometric = [&](int64_t e) { kvs_setting g = settings[e]; g.family = KVS_GBA; g.tau = 0; g.k = 0; return g; };
  kvs_setting last = as_geometric(0);
  geo[0] = last;
  if (in_brief) geo[0].family = KVS_SETTINGS_BRIEF;
  for (int64_t e = 0; e < P; ++e) {
    const kvs_setting g = as_geometric(e);
    if (e == 0 || !like(g, last, I)) {
      if ((rc = check_settings(ctx, inst, &g, 1)) != KVS_OK) return rc;
      if (e > 0 && in_brief) {                       // in full after all
        in_brief = false;
        for (int64_t x = 0; x < e; ++x) geo[x] = as_geometric(x);
      }
    }
    if (in_brief) brief[e] = make_int2(static_cast<int>(g.instance), static_cast<int>(g.M)); else geo[e] = g;
    if (e == 0 || g.instance != last.instance || length >= longest) { runs[2 * n_runs] = e; ++n_runs; length = 0; }
    runs[2 * n_runs - 1] = ++length;
    last = g;
  }
  ce = kvs_launch_bounds(inst->job_off, inst->s, inst->o, max_n, reinterpret_cast<InstStats*>(ws + L.stats), geo, P, runs, n_runs, *out,
                         reinterpret_cast<u32*>(ws + L.class_counts), ctx->stream);
  const cudaError_t marked = mark_stage(stg, ctx->stream);   // also after a failure: one of the two kernels may be running
  if (ce == cudaSuccess) ce = marked;
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "bounds launch");
  return KVS_OK;
}

static int sweep(kvs_ctx* ctx, const kvs_instances* inst, const kvs_sweep_params* params, const kvs_sweep_out* out) {
  int rc = check_instances(ctx, inst);
  if (rc) return rc;
  if (!params || !out) return fail(ctx, KVS_E_ARG, "sweep: params or out is null");
  if (inst->o_est || inst->window != 0) return fail(ctx, KVS_E_ARG, "sweep: needs offline instances ordered by the exact response length");
  if (params->instance < 0 || params->instance >= inst->n_instances) return fail(ctx, KVS_E_ARG, "sweep: instance out of range");
  if (params->family == KVS_GBA || params->family == KVS_GSA) {
    // one evaluation per initial slice, through the fused path, scalars only
    if (params->n_beta0 < 0 || params->n_beta0 > 65536) return fail(ctx, KVS_E_RANGE, "sweep: more than 65536 initial slices");
    if (params->n_beta0 == 0) return KVS_OK;
    if (!params->beta0) return fail(ctx, KVS_E_ARG, "sweep: null grid");
    const int64_t P = params->n_beta0;
    std::vector<kvs_setting> st(static_cast<size_t>(P));
    for (int64_t i = 0; i < P; ++i) {
      kvs_setting& s = st[static_cast<size_t>(i)];
      s = kvs_setting{};
      s.instance = params->instance; s.family = params->family; s.alpha_num = params->alpha_num; s.alpha_den = params->alpha_den;
      s.s_bar = -1; s.M = params->M; s.beta0 = params->beta0[i]; s.subroutine = params->subroutine; s.per_class_s = params->per_class_s;
    }
    const Layout L = make_layout(inst->n_jobs_total, inst->n_instances, inst->max_jobs_per_instance, P, false);
    if (L.total > ctx->workspace_bytes) return fail(ctx, KVS_E_CAPACITY, "workspace too small for the sweep (see kvs_workspace_bytes)");
    kvs_eval_out ev{};
    ev.peak = out->peak; ev.flow = out->flow; ev.horizon = out->horizon; ev.job_steps = out->job_steps; ev.feasible = out->feasible;
    ev.n_unfinished = reinterpret_cast<int64_t*>(ctx->workspace + L.sweep_unf);
    ev.status = reinterpret_cast<int32_t*>(ctx->workspace + L.sweep_stat);
    rc = run_fused(ctx, inst, st.data(), P, nullptr, &ev, 1);
    if (rc) return rc;
    if (out->n_completed) {
      const cudaError_t ce = kvs_launch_completed(inst->job_off + params->instance, ev.n_unfinished, ev.status, out->n_completed, P, ctx->stream);
      if (ce != cudaSuccess) return fail_cuda(ctx, ce, "sweep launch");
    }
    return KVS_OK;
  }
  if (params->family != KVS_SPS && params->family != KVS_SIMS) return fail(ctx, KVS_E_ARG, "sweep: unknown family");
  if (params->n_tau < 0 || params->n_k < 0 || static_cast<int64_t>(params->n_tau) * params->n_k > 65536)
    return fail(ctx, KVS_E_RANGE, "sweep: grid larger than 65536 settings");
  if (params->n_tau == 0 || params->n_k == 0) return KVS_OK;
  if (!params->tau || !params->k) return fail(ctx, KVS_E_ARG, "sweep: null grid");
  if (params->M < 1 || params->M >= KVS_TIME_LIMIT) return fail(ctx, KVS_E_RANGE, "sweep: M outside [1, 2^31)");
  for (int i = 0; i < params->n_tau; ++i)
    if (params->tau[i] < 1 || params->tau[i] >= KVS_TIME_LIMIT) return fail(ctx, KVS_E_RANGE, "sweep: tau outside [1, 2^31)");
  for (int i = 0; i < params->n_k; ++i)
    if (params->k[i] < 1 || params->k[i] >= KVS_TIME_LIMIT) return fail(ctx, KVS_E_RANGE, "sweep: k outside [1, 2^31)");
  const int64_t N = inst->n_jobs_total, max_n = inst->max_jobs_per_instance;
  const SweepLayout L = make_sweep_layout(max_n);
  if (L.total > ctx->workspace_bytes) return fail(ctx, KVS_E_CAPACITY, "workspace too small for the sweep (see kvs_workspace_bytes)");
  cudaError_t ce = cudaSetDevice(ctx->device);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "cudaSetDevice");
  unsigned char* ws = ctx->workspace;

  // The instance's range and its largest response are device values: one read (32 bytes, through pinned memory)
  // sizes the launches below and checks the range against the stated sizes.
  OrderInfo* const info_dev = reinterpret_cast<OrderInfo*>(ws + L.info);
  if (!ctx->pinned && (ce = cudaMallocHost(&ctx->pinned, 256)) != cudaSuccess) return fail_cuda(ctx, ce, "cudaMallocHost");
  OrderInfo* const info = static_cast<OrderInfo*>(ctx->pinned);
  ce = kvs_launch_order_info(inst->job_off + params->instance, inst->s, inst->o, N, max_n, info_dev, ctx->sm_count, ctx->stream);
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(info, info_dev, sizeof(OrderInfo), cudaMemcpyDeviceToHost, ctx->stream);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(ctx->stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "read of job_off");
  const int64_t lo = info->lo, n = info->hi - info->lo;
  if (lo < 0 || n < 0 || n > max_n || lo + n > N) return fail(ctx, KVS_E_ARG, "sweep: job_off inconsistent with the stated sizes");

  int32_t* const sorted_s = reinterpret_cast<int32_t*>(ws + L.sorted_s);
  int32_t* const sorted_o = reinterpret_cast<int32_t*>(ws + L.sorted_o);
  i64* ps = reinterpret_cast<i64*>(ws + L.prefix_s);
  u32* ps32 = reinterpret_cast<u32*>(ws + L.prefix_s32);
  i64* po = reinterpret_cast<i64*>(ws + L.prefix_o);
  ce = kvs_launch_order(inst->s + lo, inst->o + lo, n, info->stats.o_max, reinterpret_cast<u64*>(ws + L.rec0), reinterpret_cast<u64*>(ws + L.rec1),
                        reinterpret_cast<u32*>(ws + L.counts), sorted_s, sorted_o, ctx->stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "sort launch");
  ce = kvs_launch_prefix(sorted_s, sorted_o, n, reinterpret_cast<i64*>(ws + L.part), ps, ps32, po, ctx->stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "prefix launch");
  kvs_ctx::Stage* stg = nullptr;
  const size_t tau_bytes = align_up(static_cast<size_t>(params->n_tau) * 8), grid_bytes = tau_bytes + static_cast<size_t>(params->n_k) * 8;
  ce = take_stage(ctx, grid_bytes, &stg);
  if (ce == cudaSuccess) {
    std::memcpy(stg->p, params->tau, static_cast<size_t>(params->n_tau) * 8);
    std::memcpy(stg->p + tau_bytes, params->k, static_cast<size_t>(params->n_k) * 8);
    ce = send_stage(stg, ws + L.grid, grid_bytes, ctx->stream);
  }
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "copy of the grids");
  SweepParams wp{};
  wp.sorted_o = sorted_o; wp.prefix_s = ps; wp.prefix_s32 = ps32; wp.prefix_o = po;
  wp.len_max = static_cast<i64>(info->stats.s_max) + info->stats.o_max;
  wp.n = n; wp.family = params->family; wp.M = params->M;
  wp.tau = reinterpret_cast<const i64*>(ws + L.grid); wp.k = reinterpret_cast<const i64*>(ws + L.grid + tau_bytes);
  wp.n_tau = params->n_tau; wp.n_k = params->n_k; wp.out = *out;
  ce = kvs_launch_sweep(wp, reinterpret_cast<i64*>(ws + L.table), ctx->stream);
  if (ce != cudaSuccess) return fail_cuda(ctx, ce, "sweep launch");
  return KVS_OK;
}

int kvs_sweep(kvs_ctx* ctx, const kvs_instances* inst, const kvs_sweep_params* params, const kvs_sweep_out* out) {
  if (!ctx) return KVS_E_STATE;
  return guarded(ctx, [&] { return sweep(ctx, inst, params, out); });
}

}  // extern "C"
