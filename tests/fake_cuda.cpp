// A CUDA runtime that runs nothing, for CPU tests of the host code of the library (csrc/kvs_api.cu): it carries out copies
// at once, gives every copy and kernel launch the memory that it reads and writes, and follows streams and events with
// vector clocks.  Two accesses to one place, one of them a write, race unless one of them is ordered before the other.
// Any call can be made to fail (`fail_at`).  The programs at the end drive the C entry points; the test builds this file with
// kvs_api.cu and runs them.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <random>
#include <string>
#include <vector>

#include "kvs_internal.cuh"
#include "kvs_spec_shape.h"

namespace {

constexpr int MAX_STREAMS = 32;
struct Clock {
  long at[MAX_STREAMS] = {};
  void join(const Clock& c) { for (int i = 0; i < MAX_STREAMS; ++i) at[i] = std::max(at[i], c.at[i]); }
};
struct Stream { int id; Clock clock; bool gone = false; };
struct Event { Clock clock; };

enum Kind { READ, WRITE, ATOMIC };
struct Access { const unsigned char* a; const unsigned char* b; Kind kind; };
struct Op { std::string name; int stream; long seq; Clock clock; std::vector<Access> acc; };

std::vector<Stream*> streams;
std::vector<Op> ops;
std::map<const unsigned char*, size_t> locked;                     // page-locked memory
Clock host;
int calls = 0, fail_at = -1, races = 0;
long news = 0, no_memory_at = -1;      // allocations of the library's host code while `library` is set, and the one that fails
bool library = false;

Stream* stream_of(cudaStream_t s) {
  if (streams.empty()) streams.push_back(new Stream{0, {}});       // the default stream
  Stream* const st = s ? reinterpret_cast<Stream*>(s) : streams[0];
  if (st->gone && races++ < 5) printf("stream %d is used after it was destroyed\n", st->id);
  return st;
}
bool fails() { return calls++ == fail_at; }
struct Outside {                       // the fake's own allocations neither count nor fail
  bool was = library;
  Outside() { library = false; }
  ~Outside() { library = was; }
};
Access span(const void* p, size_t bytes, Kind kind) {
  const unsigned char* a = static_cast<const unsigned char*>(p);
  return Access{a, a ? a + bytes : a, kind};
}
void submit(const char* name, cudaStream_t s, std::vector<Access> acc) {
  Outside outside;
  Stream* st = stream_of(s);
  st->clock.join(host);
  const long seq = ++st->clock.at[st->id];
  // places that touch or overlap become one
  std::sort(acc.begin(), acc.end(), [](const Access& x, const Access& y) { return x.kind != y.kind ? x.kind < y.kind : x.a < y.a; });
  size_t n = 0;
  for (const Access& x : acc) {
    if (x.a == x.b) continue;
    if (n && acc[n - 1].kind == x.kind && x.a <= acc[n - 1].b) acc[n - 1].b = std::max(acc[n - 1].b, x.b);
    else acc[n++] = x;
  }
  acc.resize(n);
  ops.push_back(Op{name, st->id, seq, st->clock, std::move(acc)});
}

bool before(const Op& x, const Clock& c) { return c.at[x.stream] >= x.seq; }
void find_races() {
  for (size_t j = 0; j < ops.size(); ++j)
    for (size_t i = 0; i < j; ++i) {
      if (before(ops[i], ops[j].clock)) continue;
      for (const Access& x : ops[i].acc)
        for (const Access& y : ops[j].acc) {
          if (x.kind == y.kind && x.kind != WRITE) continue;
          if (x.a < y.b && y.a < x.b) {
            if (races++ < 5) printf("race: %s on stream %d and %s on stream %d share %zu bytes\n", ops[i].name.c_str(), ops[i].stream,
                                    ops[j].name.c_str(), ops[j].stream, static_cast<size_t>(std::min(x.b, y.b) - std::max(x.a, y.a)));
          }
        }
    }
}
int outstanding(const Clock& c) {
  int n = 0;
  for (const Op& o : ops) n += before(o, c) ? 0 : 1;
  return n;
}

}  // namespace

void* operator new(size_t n) {
  if (library && news++ == no_memory_at) throw std::bad_alloc();
  if (void* p = malloc(n ? n : 1)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

// ---- the runtime ------------------------------------------------------------------------------------------------

extern "C" {
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return fails() ? cudaErrorUnknown : cudaSuccess; }
cudaError_t cudaGetDeviceProperties_v2(cudaDeviceProp* p, int) { memset(p, 0, sizeof *p); p->multiProcessorCount = 148; return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest) { *least = 0; *greatest = -5; return fails() ? cudaErrorUnknown : cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  Outside outside;
  if (fails()) return cudaErrorUnknown;
  stream_of(nullptr);
  if (streams.size() >= MAX_STREAMS) { printf("more than %d streams\n", MAX_STREAMS); exit(2); }
  streams.push_back(new Stream{static_cast<int>(streams.size()), {}});
  *s = reinterpret_cast<cudaStream_t>(streams.back());
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned f, int) { return cudaStreamCreateWithFlags(s, f); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { stream_of(s)->gone = true; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { host.join(stream_of(s)->clock); return fails() ? cudaErrorUnknown : cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { for (Stream* s : streams) host.join(s->clock); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  if (fails() || !e) return cudaErrorUnknown;
  stream_of(s)->clock.join(reinterpret_cast<Event*>(e)->clock);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  Outside outside;
  if (fails()) return cudaErrorUnknown;
  *e = reinterpret_cast<cudaEvent_t>(new Event{});
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  if (fails() || !e) return cudaErrorUnknown;
  Stream* st = stream_of(s);
  st->clock.join(host);
  reinterpret_cast<Event*>(e)->clock = st->clock;
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { host.join(reinterpret_cast<Event*>(e)->clock); return fails() ? cudaErrorUnknown : cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) {
  Outside outside;
  if (fails()) return cudaErrorUnknown;
  *p = calloc(1, n);
  locked[static_cast<unsigned char*>(*p)] = n;
  return cudaSuccess;
}
// Memory that is given back is in no operation that the host has not waited for.
cudaError_t cudaFreeHost(void* p) {
  Outside outside;
  const unsigned char* a = static_cast<const unsigned char*>(p);
  const unsigned char* b = a + locked[a];
  for (const Op& o : ops)
    for (const Access& x : o.acc)
      if (x.a < b && a < x.b && !before(o, host) && races++ < 5) printf("%s on stream %d is in flight where page-locked memory is given back\n", o.name.c_str(), o.stream);
  locked.erase(a);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind, cudaStream_t s) {
  Outside outside;
  if (fails()) return cudaErrorUnknown;
  memcpy(dst, src, n);
  submit("copy", s, {span(dst, n, WRITE), span(src, n, READ)});
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind k) {
  const cudaError_t e = cudaMemcpyAsync(dst, src, n, k, nullptr);
  return e != cudaSuccess ? e : cudaStreamSynchronize(nullptr);
}
cudaError_t cudaMemsetAsync(void* dst, int v, size_t n, cudaStream_t s) {
  Outside outside;
  if (fails()) return cudaErrorUnknown;
  memset(dst, v, n);
  submit("memset", s, {span(dst, n, WRITE)});
  return cudaSuccess;
}
}  // extern "C"

// ---- the kernels: what they read and write ------------------------------------------------------------------------

cudaError_t kvs_setup_sort() { return cudaSuccess; }
cudaError_t kvs_setup_generic() { return cudaSuccess; }
cudaError_t kvs_setup_bounds() { return cudaSuccess; }
cudaError_t kvs_setup_spec() { return cudaSuccess; }
int kvs_build_ctas_per_sm() { return 2; }
int kvs_fused_ctas_per_sm(int light) { return light ? 3 : 2; }
i64 kvs_spec_warp_bytes(i64 n) { return 64 * (n + 64); }
i64 kvs_order_chunks(i64 n) { return n / 4096 + 1; }
i64 kvs_sweep_blocks(i64 n) { return n / 64 + 1; }
cudaError_t kvs_fused_check_word(unsigned long long*, int*, int) { return cudaSuccess; }
cudaError_t kvs_refill_check_word(unsigned long long*, int*, int) { return cudaSuccess; }
cudaError_t kvs_spec_check_word(unsigned long long*, int*, int) { return cudaSuccess; }

cudaError_t kvs_launch_sort(const SortParams& p, int, cudaStream_t s) {
  Outside outside;
  if (fails()) return cudaErrorUnknown;
  const i64 lo = p.job_off[0], n = p.job_off[p.n_instances] - lo;
  std::vector<Access> a = {span(p.job_off, 8 * (p.n_instances + 1), READ), span(p.s + lo, 4 * n, READ), span(p.o + lo, 4 * n, READ),
                           span(p.stats, sizeof(InstStats) * p.n_instances, WRITE)};
  for (int32_t* w : {p.perm, p.perm_tmp, p.iperm, p.sorted_s, p.sorted_o}) a.push_back(span(w + lo, 4 * n, WRITE));
  submit("ordering", s, a);
  return cudaSuccess;
}

namespace {
void evaluations(const BuildParams& p, int grid, i64 e, std::vector<Access>* a) {
  const kvs_setting& st = p.settings[e];
  const i64 lo = p.job_off[st.instance], n = p.job_off[st.instance + 1] - lo;
  for (const int32_t* r : {p.sorted_s, p.sorted_o, p.iperm, p.s, p.o}) a->push_back(span(r + lo, 4 * n, READ));
  a->push_back(span(p.stats + st.instance, sizeof(InstStats), READ));
  for (i64* w : {p.ev.peak, p.ev.flow, p.ev.job_steps, p.ev.horizon, p.ev.n_unfinished})
    if (w) a->push_back(span(w + e, 8, WRITE));
  if (p.ev.status) a->push_back(span(p.ev.status + e, 4, WRITE));
}
void scratch(const BuildParams& p, int grid, std::vector<Access>* a) {
  a->push_back(span(p.lists, static_cast<size_t>(grid) * KVS_CTA_SCRATCH(p.max_jobs), WRITE));
  a->push_back(span(p.fin_rank, static_cast<size_t>(grid) * p.max_jobs * 4, WRITE));
  a->push_back(span(p.counter, 8, WRITE));
  a->push_back(span(p.settings, sizeof(kvs_setting) * p.P, READ));
}
}  // namespace

cudaError_t kvs_launch_fused(const BuildParams& p, int grid, int light, int fam, cudaStream_t s) {
  Outside outside;
  if (fails()) return cudaErrorUnknown;
  std::vector<Access> a;
  scratch(p, grid, &a);
  for (ull i = 0; i < *p.eval_count; ++i) evaluations(p, grid, p.eval_list[i], &a);
  a.push_back(span(p.slow_list, 8 * p.P, ATOMIC));
  a.push_back(span(p.slow_count, 8, ATOMIC));
  submit(light ? "light kernel" : "full kernel", s, a);
  return cudaSuccess;
}
cudaError_t kvs_launch_build(const BuildParams& p, int grid, cudaStream_t s) {
  Outside outside;
  if (fails()) return cudaErrorUnknown;
  std::vector<Access> a;
  scratch(p, grid, &a);
  for (i64 e = 0; e < p.P; ++e) evaluations(p, grid, e, &a);
  if (p.slow_list) { a.push_back(span(p.slow_list, 8 * p.P, READ)); a.push_back(span(p.slow_count, 8, READ)); }
  submit("general kernel", s, a);
  return cudaSuccess;
}
static cudaError_t unused() { printf("a launch that these tests do not drive\n"); exit(2); }
cudaError_t kvs_launch_refill(const RefillParams&, cudaStream_t) { return unused(); }
SpecParams spec_launched;
std::vector<i64> spec_groups_launched;
cudaError_t kvs_launch_spec(SpecParams p, cudaStream_t) {
  Outside outside;
  spec_launched = p;
  spec_groups_launched.assign(p.groups, p.groups + KVS_SPEC_GROUP * p.n_groups);
  return cudaSuccess;
}
cudaError_t kvs_launch_generic_tiled(GenericParams, i64, int, cudaStream_t) { return unused(); }
cudaError_t kvs_launch_bounds(const i64*, const int32_t*, const int32_t*, i64, InstStats*, const kvs_setting*, i64, const i64*, i64, const kvs_bounds_out&, u32*, cudaStream_t) { return unused(); }
cudaError_t kvs_launch_order_info(const i64*, const int32_t*, const int32_t*, i64, i64, OrderInfo*, int, cudaStream_t) { return unused(); }
cudaError_t kvs_launch_order(const int32_t*, const int32_t*, i64, int, u64*, u64*, u32*, int32_t*, int32_t*, cudaStream_t) { return unused(); }
cudaError_t kvs_launch_prefix(const int32_t*, const int32_t*, i64, i64*, i64*, u32*, i64*, cudaStream_t) { return unused(); }
cudaError_t kvs_launch_sweep(const SweepParams&, i64*, cudaStream_t) { return unused(); }
cudaError_t kvs_launch_completed(const i64*, const i64*, const int32_t*, i64*, i64, cudaStream_t) { return unused(); }

// ---- the calls ----------------------------------------------------------------------------------------------------

namespace {

constexpr int JOBS = 4;               // jobs per instance
struct Batch {
  int I;
  std::vector<i64> off;
  std::vector<int32_t> s, o;
  std::vector<kvs_setting> st;
  explicit Batch(int n_inst) : I(n_inst) {
    for (int i = 0; i <= I; ++i) off.push_back(static_cast<i64>(i) * JOBS);
    s.assign(static_cast<size_t>(I) * JOBS, 3);
    o.assign(static_cast<size_t>(I) * JOBS, 5);
  }
  void add(int inst, int family) {
    kvs_setting x{};
    x.instance = inst; x.family = family; x.alpha_num = 2; x.alpha_den = 1; x.s_bar = -1; x.M = 1000;
    st.push_back(x);
  }
};

struct Caller {
  kvs_ctx* ctx = nullptr;
  std::vector<unsigned char> memory;
  unsigned char* ws = nullptr;
  explicit Caller(int I, i64 P, uint64_t need = 0) {
    ops.clear();
    streams.clear();
    host = Clock{};
    if (!need) kvs_workspace_bytes(static_cast<i64>(I) * JOBS, I, JOBS, P, 0, 1, &need);
    memory.resize(need + 512);
    ws = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(memory.data()) + 255) & ~static_cast<uintptr_t>(255));
    kvs_init_params prm{};
    prm.workspace = ws; prm.workspace_bytes = need;
    if (kvs_init(&prm, &ctx) != KVS_OK) { printf("kvs_init failed\n"); exit(2); }
  }
  ~Caller() { kvs_destroy(ctx); }
};

kvs_instances view(const Batch& b) {
  kvs_instances in{};
  in.n_instances = b.I; in.n_jobs_total = static_cast<i64>(b.I) * JOBS; in.max_jobs_per_instance = JOBS;
  in.job_off = b.off.data(); in.s = b.s.data(); in.o = b.o.data();
  return in;
}

int host_call(Caller& c, const Batch& b) {
  const size_t P = b.st.size();
  std::vector<i64> peak(P), flow(P);
  std::vector<int32_t> status(P);
  kvs_eval_out ev{};
  ev.peak = peak.data(); ev.flow = flow.data(); ev.status = status.data();
  const kvs_instances in = view(b);
  library = true;
  const int rc = kvs_evaluate_built_host(c.ctx, &in, b.st.data(), static_cast<i64>(P), &ev);
  library = false;
  return rc;
}
int device_call(Caller& c, const Batch& b) {
  std::vector<i64> peak(b.st.size());
  kvs_eval_out ev{};
  ev.peak = peak.data();
  const kvs_instances in = view(b);
  library = true;
  const int rc = kvs_evaluate_built(c.ctx, &in, b.st.data(), static_cast<i64>(b.st.size()), nullptr, &ev);
  library = false;
  return rc;
}

// What a program does that does not know its sizes: they are read and the offsets formed, then the call is made.
int sized_call(Caller& c, kvs_reader* r, const Batch& b) {
  const i64 P = static_cast<i64>(b.st.size());
  std::vector<i64> cap, offsets(2 * static_cast<size_t>(P) + 2);
  for (i64 e = 0; e < P; ++e) cap.push_back(e % 7);
  i64 *const job_off = offsets.data(), *const prof_off = job_off + P + 1;
  kvs_sizes sizes{};
  library = true;
  int rc = kvs_sizes_begin(r, nullptr, b.off.data(), b.I, cap.data(), P);
  if (rc == KVS_OK) rc = kvs_sizes_end(r, b.st.data(), P, job_off, prof_off, &sizes);
  library = false;
  if (rc != KVS_OK) return rc;
  i64 jobs = 0, rounds = 0;
  for (i64 e = 0; e < P; ++e) {
    const i64 inst = b.st[static_cast<size_t>(e)].instance;
    if (job_off[e] != jobs || prof_off[e] != rounds) { printf("offsets of evaluation %ld: %ld, %ld\n", static_cast<long>(e), static_cast<long>(job_off[e]), static_cast<long>(prof_off[e])); ++races; break; }
    jobs += b.off[static_cast<size_t>(inst) + 1] - b.off[static_cast<size_t>(inst)];
    rounds += cap[static_cast<size_t>(e)];
  }
  if (sizes.max_jobs != JOBS || sizes.job_results != jobs || sizes.profile_rounds != rounds) { printf("wrong sizes\n"); ++races; }
  std::vector<int32_t> start(static_cast<size_t>(jobs)), done(start.size());
  std::vector<i64> peak(static_cast<size_t>(P));
  kvs_schedule_out out{};
  out.job_out_off = job_off; out.job_start = start.data(); out.job_completion = done.data();
  kvs_eval_out ev{};
  ev.peak = peak.data();
  const kvs_instances in = view(b);
  library = true;
  rc = kvs_evaluate_built(c.ctx, &in, b.st.data(), P, &out, &ev);
  library = false;
  return rc;
}

void run_host(const char* name, const Batch& b) {
  Caller c(b.I, static_cast<i64>(b.st.size()));
  const int r0 = races;
  for (int twice = 0; twice < 2; ++twice)
    if (const int rc = host_call(c, b)) { printf("%s: status %d\n", name, rc); ++races; }
  find_races();
  if (const int n = outstanding(host)) { printf("%s: %d operations in flight after the call\n", name, n); ++races; }
  if (races != r0) printf("%s: %d\n", name, races - r0);
}

// chunks of unequal size, chunks of unequal composition, calls that do and do not split by family
void overlaps() {
  for (int I : {1024, 1000, 900, 769}) {
    Batch b(I);
    for (int i = 0; i < I; ++i) for (int f = KVS_GBA; f <= KVS_SIMS; ++f) b.add(i, f);
    run_host(("four families on " + std::to_string(I)).c_str(), b);
  }
  std::mt19937 rng(7);
  for (int rep = 0; rep < 8; ++rep) {
    const int I = 600 + static_cast<int>(rng() % 700);
    Batch b(I);
    for (int i = 0; i < I; ++i) {
      // later instances: more evaluations of the light variant, single families, or many of the full one
      const int more = rep % 3 == 0 ? 1 + 6 * i / I : 2;
      b.add(i, KVS_GSA);
      for (int k = 0; k < more; ++k) b.add(i, rep % 4 == 0 ? KVS_SPS : static_cast<int>(rng() % 4));
      if (rep % 3 == 2 && i > I / 2) for (int k = 0; k < 5; ++k) b.add(i, KVS_GSA);
    }
    if (rep % 2) std::shuffle(b.st.begin(), b.st.end(), rng);
    run_host(("mixture " + std::to_string(rep)).c_str(), b);
  }
}

// Requests for sizes: several at a time on readers of their own, one at a time on one reader, sizes that grow, readers on two streams.
void sizes() {
  Caller c(1, 1);
  auto expect = [&](const char* what, bool ok) { if (!ok) { printf("%s\n", what); ++races; } };
  kvs_reader *x = nullptr, *y = nullptr;
  expect("open", kvs_reader_open(0, &x) == KVS_OK && kvs_reader_open(0, &y) == KVS_OK && kvs_reader_open(1, nullptr) == KVS_E_ARG);
  const std::vector<i64> a = {0, 3, 7}, b = {0, 50, 90}, cap = {11, 0};
  kvs_setting st[2]{};
  st[1].instance = 1;
  kvs_sizes sa{}, sb{};
  std::vector<i64> oa(3), ob(3), pa(3);
  // interleaved: each end is that of its own begin
  expect("begin", kvs_sizes_begin(x, nullptr, a.data(), 2, cap.data(), 2) == KVS_OK && kvs_sizes_begin(y, nullptr, b.data(), 2, nullptr, 0) == KVS_OK);
  expect("a second begin is refused", kvs_sizes_begin(x, nullptr, b.data(), 2, nullptr, 0) == KVS_E_STATE && kvs_reader_error(x)[0] != 0);
  expect("end", kvs_sizes_end(x, st, 2, oa.data(), pa.data(), &sa) == KVS_OK && kvs_sizes_end(y, st, 2, ob.data(), nullptr, &sb) == KVS_OK);
  expect("sizes of the first", sa.max_jobs == 4 && sa.job_results == 7 && sa.profile_rounds == 11 && oa == a && pa == std::vector<i64>({0, 11, 11}));
  expect("sizes of the second", sb.max_jobs == 50 && sb.job_results == 90 && sb.profile_rounds == 0 && ob == b);
  expect("an end without a begin is refused", kvs_sizes_end(x, st, 2, oa.data(), nullptr, &sa) == KVS_E_STATE);
  // a request that is refused at its end is over
  st[1].instance = 2;
  kvs_sizes_begin(x, nullptr, a.data(), 2, nullptr, 0);
  expect("instance out of range", kvs_sizes_end(x, st, 2, oa.data(), nullptr, &sa) == KVS_E_ARG);
  kvs_sizes_begin(x, nullptr, a.data(), 2, nullptr, 0);
  expect("capacities that were not asked for", kvs_sizes_end(x, st, 2, nullptr, pa.data(), &sa) == KVS_E_ARG);
  expect("the next request", kvs_sizes_begin(x, nullptr, a.data(), 2, nullptr, 0) == KVS_OK && kvs_sizes_end(x, st, 1, oa.data(), nullptr, &sa) == KVS_OK && oa[1] == 3);
  // sizes below zero: none of the offsets precedes the one before it
  const std::vector<i64> negative = {5, -1}, falling = {0, 4, 1, 3};
  kvs_sizes_begin(x, nullptr, nullptr, 0, negative.data(), 2);
  expect("a negative capacity is refused", kvs_sizes_end(x, nullptr, 2, nullptr, pa.data(), &sa) == KVS_E_ARG);
  kvs_setting three[3]{};
  for (int i = 0; i < 3; ++i) three[i].instance = i;
  std::vector<i64> of(4);
  kvs_sizes_begin(x, nullptr, falling.data(), 3, nullptr, 0);
  expect("falling offsets", kvs_sizes_end(x, three, 3, of.data(), nullptr, &sa) == KVS_OK && of == std::vector<i64>({0, 4, 4, 6}) && sa.max_jobs == 4);
  // requests of growing size under two streams in turn: what one uploads is not overwritten by the next
  cudaStream_t other = nullptr;
  cudaStreamCreateWithFlags(&other, 0);
  std::vector<std::vector<i64>> keep;
  for (int i = 1; i < 6; ++i) {
    const size_t P = static_cast<size_t>(200) << (2 * i);
    keep.emplace_back(P, 3);
    keep.emplace_back(P + 1, 0);
    expect("a request", kvs_sizes_begin(x, i % 2 ? other : nullptr, nullptr, 0, keep[keep.size() - 2].data(), static_cast<i64>(P)) == KVS_OK &&
                            kvs_sizes_end(x, nullptr, static_cast<i64>(P), nullptr, keep.back().data(), &sa) == KVS_OK && sa.profile_rounds == 3 * static_cast<i64>(P));
  }
  find_races();
  // a request that is never ended, on a stream that its caller destroys: the reader waits for the copy, not on the stream
  kvs_sizes_begin(y, other, b.data(), 2, nullptr, 0);
  cudaStreamDestroy(other);
  kvs_reader_close(y);
  kvs_reader_close(x);
  if (const int n = outstanding(host)) { printf("%d operations in flight\n", n); ++races; }
}

// How a call's speculative runs are laid out: on which kernel, how many evaluations of an SM are in flight, groups of one instance
// that hold every evaluation once.  `most`: evaluations of one instance that a CTA takes (0: none, all in memory); `live`: per SM.
void spec_call(int jobs, const std::vector<int>& evals_of, int most, double live) {
  const int r0 = races;
  Batch b(static_cast<int>(evals_of.size()));
  for (size_t i = 0; i < evals_of.size(); ++i)
    for (int k = 0; k < evals_of[i]; ++k) { b.add(static_cast<int>(i), KVS_GSAS); b.st.back().M = 1000 + (7 * k + static_cast<int>(i)) % 50; }
  const i64 P = static_cast<i64>(b.st.size());
  uint64_t need = 0;
  kvs_workspace_bytes(static_cast<i64>(b.I) * JOBS, b.I, jobs, P, 0, 1, &need);
  Caller c(b.I, P, need);
  kvs_instances in = view(b);
  in.max_jobs_per_instance = jobs;
  std::vector<i64> off(static_cast<size_t>(P) + 1, 0), peak(static_cast<size_t>(P)), horizon(peak.size());
  std::vector<int32_t> out(1), status(peak.size());
  alignas(16) static int32_t profile[4];
  kvs_schedule_out so{};
  so.job_out_off = off.data(); so.job_start = out.data(); so.job_completion = out.data();
  kvs_eval_out ev{};
  ev.profile_off = off.data(); ev.profile = profile; ev.peak = peak.data(); ev.horizon = horizon.data(); ev.status = status.data();
  if (const int rc = kvs_evaluate_built(c.ctx, &in, b.st.data(), P, &so, &ev)) { printf("status %d\n", rc); ++races; return; }
  const SpecParams& p = spec_launched;
  std::vector<int> seen(static_cast<size_t>(P), 0);
  i64 last = 0;
  for (i64 g = 0; g < p.n_groups; ++g) {
    const i64* e = spec_groups_launched.data() + KVS_SPEC_GROUP * g;
    const kvs_setting& first = b.st[static_cast<size_t>(e[0])];
    const i64 in_all = evals_of[static_cast<size_t>(first.instance)], least = in_all / spec_groups(in_all, p.group_warps);
    i64 size = 0, budget = 0;
    for (int i = 0; i < KVS_SPEC_GROUP; ++i) {
      if (e[i] < 0) continue;
      const kvs_setting& st = b.st[static_cast<size_t>(e[i])];
      if (i != size++ || st.instance != first.instance || st.M < budget) { printf("group %ld\n", static_cast<long>(g)); ++races; }
      budget = st.M;
      ++seen[static_cast<size_t>(e[i])];
    }
    if (size > p.group_warps || size < least || size > least + 1 || first.M < last) { printf("group %ld: %ld evaluations\n", static_cast<long>(g), static_cast<long>(size)); ++races; }
    last = first.M;
  }
  if (p.n_groups && std::count(seen.begin(), seen.end(), 1) != P) { printf("an evaluation is missing\n"); ++races; }
  const i64 held = p.n_groups ? 148l * spec_resident(jobs, p.group_warps, p.ring) : 0;
  const double found = p.n_groups ? static_cast<double>(P) / 148 * std::min(1.0, static_cast<double>(held) / static_cast<double>(p.n_groups)) : 0.0;
  if (p.n_groups && (spec_cta_bytes(jobs, p.group_warps, p.ring) > 227 * 1024 || p.ring & (p.ring - 1) || p.ring < 256)) { printf("CTA\n"); ++races; }
  if ((p.n_groups ? p.group_warps : 0) != most || found < live - 0.01) { printf("%d per CTA, %.2f per SM\n", p.n_groups ? p.group_warps : 0, found); ++races; }
  if (races != r0) printf("jobs %d, %ld evaluations\n", jobs, static_cast<long>(P));
}
void groups() {
  auto each = [](int instances, int evals) { return std::vector<int>(static_cast<size_t>(instances), evals); };
  // one budget per instance: no CTA holds room for more than it has
  for (int P : {1, 512, 2048, 8192}) {
    spec_call(500, each(P, 1), 1, std::min(16.0, P / 148.0));
    spec_call(5000, each(P, 1), 1, std::min(4.0, P / 148.0));
  }
  spec_call(10000, each(2048, 1), 1, 2.0);
  // five: three and two, or none of them waits for a place
  spec_call(10000, each(410, 5), 3, 2.5);
  spec_call(5000, each(1639, 5), 2, 5.0);
  spec_call(500, each(13, 5), 3, 0.43);
  // eight: as many as an SM holds
  spec_call(10000, each(64, 8), 4, 3.45);
  spec_call(10000, each(1024, 8), 4, 4.0);
  spec_call(5000, each(1024, 8), 2, 6.0);
  spec_call(16000, each(256, 8), 2, 2.0);
  // instances with different numbers of them; some with none
  std::vector<int> mixed;
  for (int i = 0; i < 300; ++i) mixed.push_back(i % 10);
  spec_call(3000, mixed, 3, 7.5);
  // more than can be in flight by far, few of them at a time: the kernel in memory; as many as that one would not win back: on chip
  spec_call(24000, each(2300, 1), 1, 1.0);
  spec_call(24000, each(2700, 1), 0, 0.0);
  spec_call(10000, each(6500, 1), 1, 2.0);
  spec_call(10000, each(8192, 1), 0, 0.0);
  // not even one fits, or 16 bits do not number the jobs
  spec_call(30000, each(10, 2), 0, 0.0);
  spec_call(65535, each(10, 2), 0, 0.0);
}

// A refused call enqueues nothing; a call that fails half-way (every fallible call of the runtime, every launch and every
// allocation in turn) returns a status and leaves nothing behind that the next call could meet.
void errors() {
  Batch b(520);
  for (int i = 0; i < b.I; ++i) for (int f = KVS_GBA; f <= KVS_SIMS; ++f) b.add(i, f);
  auto next_call = [&](const char* name, Caller& c) {
    if (host_call(c, b) != KVS_OK) { printf("%s: the next call fails\n", name); ++races; }
    find_races();
  };
  for (int family : {KVS_GBAD, KVS_GSAS}) {
    Batch bad = b;
    bad.st.back().family = family;
    Caller c(b.I, static_cast<i64>(b.st.size()));
    if (host_call(c, bad) != KVS_E_ARG || !ops.empty()) { printf("family %d: %zu operations of a refused call\n", family, ops.size()); ++races; }
    next_call("refused", c);
  }
  enum { HOST, DEVICE, SIZED };
  for (bool memory : {false, true})
    for (int kind : {HOST, DEVICE, SIZED}) {
      const bool device = kind != HOST;
      int rc = KVS_E_CUDA, n = 0;
      for (; rc != KVS_OK && n < 2000; ++n) {
        Caller c(b.I, static_cast<i64>(b.st.size()));
        kvs_reader* r = nullptr;
        if (kvs_reader_open(0, &r) != KVS_OK) { printf("kvs_reader_open failed\n"); exit(2); }
        calls = 0;
        news = 0;
        no_memory_at = memory ? n : -1;
        fail_at = memory ? -1 : n;
        rc = kind == SIZED ? sized_call(c, r, b) : (device ? device_call(c, b) : host_call(c, b));
        fail_at = -1;
        no_memory_at = -1;
        if (rc != KVS_OK && rc != (memory ? KVS_E_STATE : KVS_E_CUDA)) { printf("status %d\n", rc); ++races; }
        // the host entry point is over when it returns; what a device one has launched precedes the stream's next work
        if (const int left = outstanding(device ? stream_of(nullptr)->clock : host)) {
          if (races++ < 5) printf("%s call, failure %d: %d operations in flight\n", device ? "device" : "host", n, left);
        }
        if (kind == SIZED) {
          // the reader is ready for another request, or is given back with its last one in flight
          if (n % 2 && sized_call(c, r, b) != KVS_OK) { printf("the reader's next request fails\n"); ++races; }
          if (n % 3 == 0) kvs_sizes_begin(r, nullptr, b.off.data(), b.I, nullptr, 0);
        }
        kvs_reader_close(r);
        next_call("after a failure", c);
      }
      const int least = memory ? (device ? 1 : 4) : (kind == SIZED ? 18 : (device ? 10 : 80));
      if (n < least || n == 2000) { printf("%d failures\n", n); ++races; }
    }
}

}  // namespace

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  if (what == "overlaps") overlaps();
  else if (what == "errors") errors();
  else if (what == "sizes") sizes();
  else if (what == "groups") groups();
  else { printf("unknown program\n"); return 2; }
  printf("%s: %d faults\n", what.c_str(), races);
  return races ? 1 : 0;
}
