// Fused schedule builder and evaluator, 32-bit fast path: one CTA per (instance, setting, family)
// evaluation, times below 2^31.
//
// For one evaluation (and one arrival window at a time) the CTA
//   1. forms the phase table: the geometric ladder tau_p with the largest memory-feasible
//      parallelism k_p (first line of the two geometric algorithms; Lemma "Peak Memory Usage of
//      SPS"; Eq. max-parallelism), or the single (tau, k) of SPS / SimS;
//   2. plans the phases without touching a run: a job enters at the class f of its key and leaves
//      at the class l of the larger of key and response length, so phase p has
//      N_p = #{f <= p} - #{l < p} participants; that fixes every phase's length
//      floor((N_p - 1) tau_p / k_p) + tau_p and first round;
//   3. writes every job's start and completion: the job's rank in the phase that completes it is
//      the number of earlier positions (in schedule order) that leave in that phase or later; for
//      exact keys that is the position inside the class, otherwise it is counted with one warp
//      ballot per phase over 32 positions at a time, behind per-warp class histograms.
//      start = base_p + floor(r*tau_p/k_p) (Procedure StaggeredPipelineSchedule) or
//      base + floor(r/k)*tau (simultaneous batches), completion = start + o;
//   4. if the memory profile is wanted, walks the phases tile by tile as the general kernel does:
//      the runs that start inside a tile are a contiguous rank range, every run adds (c, 1) at its
//      first round and (-c, -1) after its last one to two shared-memory difference arrays
//      (c = s + 1 - start), one scan per array gives memory(t) = A(t) + t*B(t)
//      (Eq. Memory-Feasibility), the peak is reduced and the profile stored 16 bytes at a time.
//      Jobs killed at the end of their slot are carried to the next phase as (s, o) pairs, so a
//      phase reads its participants as one contiguous stream;
//   5. if only the peak is wanted, walks rounds as the last resort.  Exact keys: one candidate per run end from prefix sums,
//      per class.  Slicing: the phases from the last one back, as slices and with them the memory held grow along the ladder;
//      a phase whose widest window of k_p ranks cannot exceed the largest memory found so far is skipped, one of few pairs of
//      runs is summed run end by run end, the rest are walked (128 instances of 10,000 jobs, eight budgets, both families:
//      1,880 us with every phase walked, 917 us).  Simultaneous batches: prefix sums, or one bucket per batch and round in
//      which one of its runs can end (64 instances of 5,000 jobs, two budgets: 716 us in the general kernel, 253 us).
//
// What bounds it: instruction issue and the latency between block barriers, not memory (slicing with a profile: about 2 M warp
// instructions per evaluation of 50,000 jobs, half of the issue slots in use, DRAM at a tenth of the copy bandwidth).
// A call of few evaluations (one per SM or fewer) gives each of them to several CTAs, see FusedShare: one evaluation of each of
// four families on one instance of 1,000 jobs took 130 us on four CTAs and 33 us on 64.
//
// An evaluation whose times reach 2^31 or whose memory bound reaches 2^32 is not finished here: its
// index is appended to a list that the general kernel works off afterwards.
#include <cstddef>

#include "kvs_events.cuh"
#include "kvs_ladder.cuh"

namespace {

constexpr int T = KVS_EVAL_THREADS;
constexpr int ITEMS = KVS_EVAL_ITEMS;
constexpr int TILE = KVS_TILE;
constexpr int WARPS = T / 32;
constexpr int VEC = ITEMS / 4;
constexpr int RPT = 4;                       // consecutive ranks per thread in the run visit
constexpr int MAXP = KVS_MAX_PHASES;
constexpr int RINGW = 2 * TILE + (2 * TILE) / 8;
constexpr int GCOL = 2049;
// What a peak without rounds is weighed by (see the uses): cycles that a step of a thread over the pairs of a run end and a run is taken to
// cost, and the pairs of a phase above which all CTAs of an evaluation look at them.  The step itself - a load, a comparison, two
// additions - costs less, but at its own cost phases went to the run ends that the bound or the visit settles sooner.  us a call of plain
// slicing on config 2's lengths, cycles 40 / 60 / 80 / 100 / 150 (2^20 pairs):
//   sweeps over 64 initial slices: 500 jobs alike, 2,000 (2^20 tokens) 125 / 103 / 101 / 101 / 106, 5,000 183 / 163 / 151 / 147 / 163, 20,000 (2^22) 361 / 337 / 316 / 319 / 319;
//   2 instances of 100,000 jobs 643 / 643 / 583 / 486 / 486, 1,024 of 20,000 from host memory 3,370 / 3,222 / 3,233 / 3,215 / 3,217.
// Pairs 2^18 / 2^19 / 2^20 / 2^21 / 2^22 / never (100 cycles):
//   sweeps: 500 jobs alike, 2,000 (16 values, 2^22) 104 / 99 / 86 / 87 / 87 / 86, 5,000 (64, 2^20) 132 / 133 / 147 / 147 / 149 / 148, (4, 2^22) 93 / 90 / 90 / 112 / 112 / 112,
//   20,000 (64, 2^18) 223 / 220 / 201 / 202 / 201 / 202, (64, 2^20) 237 / 240 / 237 / 296 / 334 / 331;  2 instances of 100,000 jobs 505 / 506 / 484 / 473 / 474 / 518.
constexpr int PAIR_CYCLES = 100;
constexpr u64 SHARED_PAIRS = 1u << 20;
static_assert((TILE & (TILE - 1)) == 0 && ITEMS % 4 == 0 && ITEMS <= 32 && 32 % ITEMS == 0, "tile layout");
constexpr u32 TIME_LIMIT = 0x7fffffffu - 4u * TILE;   // phase ends stay below this

// Checked build (-DKVS_DEBUG): every computed index into the ring, the per-CTA scratch (class bytes, rank
// table, lists, start rounds, prefix sums) and the caller's profile and per-job outputs is tested against
// its bound before the access.  A violation records (code << 56 | index) in one device word - the first
// one wins - and the access is skipped; nothing traps.  The host reads the word with
// kvs_debug_check_word.  In the normal build KVS_IN is the constant true and costs nothing.
#ifdef KVS_DEBUG
__device__ unsigned long long g_check_word = 0ull;
__device__ __forceinline__ bool kvs_in_range(i64 idx, i64 limit, int code) {
  if (idx >= 0 && idx < limit) return true;
  atomicCAS(&g_check_word, 0ull, (static_cast<ull>(code) << 56) | (static_cast<ull>(idx) & 0x00ffffffffffffffull));
  return false;
}
#define KVS_IN(idx, limit, code) kvs_in_range(static_cast<i64>(idx), static_cast<i64>(limit), (code))
#else
#define KVS_IN(idx, limit, code) true
#endif
enum { CHK_GCOL = 1, CHK_G = 2, CHK_CLS = 3, CHK_RING = 4, CHK_LIST = 5, CHK_LIST_OUT = 6, CHK_PS = 7, CHK_PROFILE = 8,
       CHK_JOB_OUT = 11, CHK_FIN = 12, CHK_Z = 13 };

struct FShared {
  u128 pw_a[MAXP + 1];
  u128 pw_b[MAXP + 1];
  u64 taupre[MAXP + 1];       // sum of tau_q over q < p
  u64 kinv[MAXP];             // floor(2^64 / k_p) + 1, see slot_mul
  i64 plen[MAXP];
  i64 red64[32];
  i64 next_eval;
  i64 base_next;
  i64 n_runs;
  u32 tau[MAXP], k[MAXP], pbase[MAXP], np[MAXP];
  u32 cnt[WARPS][MAXP];       // per-warp class counts, then ranks before each warp's segment
  u32 gcol[GCOL];             // the current phase's column of the rank table (windows of up to (GCOL-1)*256 jobs)
  u32 redA[32], redB[32];
  int red32[32];
  int ent[MAXP + 1];          // class boundaries in key order
  int n_phases, seg_end, fallback;
  u32 s_top[MAXP];            // longest prompt per class
  int tile_lo[MAXP], tile_hi[MAXP];   // tiles of every phase that this CTA walks (evaluations shared by several CTAs)
  // two-tile ring of difference arrays: constant terms and slopes.  Round e of the ring (0 <= e <
  // 2*TILE) lives at word e + 4*(e/32): four spare words after every 32 keep the 16-byte loads of
  // the scan (a thread owns ITEMS consecutive rounds) free of bank conflicts while the index of an
  // event stays a shift and an add.  Last in the struct: the kernel for evaluations that walk no
  // rounds is launched without this part.
  alignas(16) u32 dA[RINGW];
  alignas(16) u32 dB[RINGW];
};

// floor(r * tau / k) for r, tau, k below 2^31 with a result below 2^31
__device__ __forceinline__ u32 slot32(u32 r, u32 tau, u32 k) {
  const u64 x = static_cast<u64>(r) * tau;
  if ((x >> 32) == 0) return static_cast<u32>(x) / k;
  return static_cast<u32>(x / k);
}

// The same with the division replaced by a multiplication: kinv = floor(2^64 / k) + 1 (k >= 2).
// For x = r * tau below 2^32, x * kinv / 2^64 = x/k + x*e/(k*2^64) with 0 < e <= k; the excess is
// below 2^-32 while the fractional part of x/k stays at least 1/k > 2^-31 short of the next integer,
// so the high word of the product is exactly floor(x / k).
__device__ __forceinline__ u32 slot_mul(u32 r, u32 tau, u32 k, u64 kinv) {
  const u64 x = static_cast<u64>(r) * tau;
  if ((x >> 32) == 0) return k == 1 ? static_cast<u32>(x) : static_cast<u32>(__umul64hi(x, kinv));
  return static_cast<u32>(x / k);
}

// Word of the round `rel` rounds after the origin of ring half `buf`, 0 <= rel < 2*TILE.
__device__ __forceinline__ int ring(int buf, int rel) {
  if (!KVS_IN(rel, 2 * TILE, CHK_RING)) rel = 0;
  const int e = (buf * TILE + rel) & (2 * TILE - 1);
  return e + ((e >> 5) << 2);
}

// One phase as the run visit sees it.  Positions are relative to the window, in schedule order.
// Exact keys: the participants are the positions [x_lo, x_hi) and the rank is the offset from x_lo.
// Carried jobs (FILTER): position x < x_hi takes part iff its leaving class cls[x] >= ph, and the
// rank table G[seg * L + ph] holds the number of such positions before segment `seg` (SEG positions
// each), so a warp can start at any segment without looking at the ones before it.
struct PhaseView {
  const int32_t* S;
  const int32_t* O;
  const unsigned char* cls;
  const u32* G;
  const u32* gcol;        // column ph of G in shared memory, or NULL
  int L, ph, nsegs;
  int cls_cap, g_cap;     // bytes of cls and words of G in this CTA's scratch
  int n_src;              // positions of the window (S and O may be read below this index)
  int x_lo, x_hi;
  u32 tau, k, qt, rt;     // tau = qt*k + rt
  u32 len;                // rounds of the phase
  u32 base;               // its first round
};

constexpr int SEG = 256;  // positions per warp step: 8 consecutive positions per lane

// participants of the phase before segment `seg`
__device__ __forceinline__ int rank_before(const PhaseView& P, int seg) {
  if (P.gcol) return KVS_IN(seg, GCOL, CHK_GCOL) ? static_cast<int>(P.gcol[seg]) : 0;
  return KVS_IN(seg * P.L + P.ph, P.g_cap, CHK_G) ? static_cast<int>(P.G[seg * P.L + P.ph]) : 0;
}

// The 8 positions of one lane in segment `seg`: bit j of `bits` is set if position xb + j takes part,
// and those positions have the consecutive ranks r_first, r_first + 1, ...
// With FILTER, `fbits` marks the participants whose leaving class is this phase (they complete here;
// the others are killed at the end of their slot and their response length is not needed).
struct LaneGroup { u32 bits; u32 fbits; int r_first; int xb; };

// Bit j of the result is set iff byte j of `w` is >= (ge) or == the byte replicated in `p4`.
__device__ __forceinline__ u32 byte_mask4(u32 w, u32 p4, bool ge) {
  const u32 m = (ge ? __vcmpgeu4(w, p4) : __vcmpeq4(w, p4)) & 0x08040201u;
  return (m | (m >> 8) | (m >> 16) | (m >> 24)) & 15u;
}

template <bool FILTER>
__device__ __forceinline__ LaneGroup lane_group(const PhaseView& P, int seg) {
  LaneGroup g;
  const int lane = lane_id();
  if (FILTER) {
    g.xb = seg * SEG + 8 * lane;
    const uint2 cw = KVS_IN(g.xb + 7, P.cls_cap, CHK_CLS) ? *reinterpret_cast<const uint2*>(P.cls + g.xb) : make_uint2(0, 0);
    const int room = P.x_hi - g.xb;                        // positions of this lane below x_hi
    const u32 lim = room >= 8 ? 0xffu : (room > 0 ? (1u << room) - 1u : 0u);
    const u32 p4 = static_cast<u32>(P.ph) * 0x01010101u;
    g.bits = (byte_mask4(cw.x, p4, true) | byte_mask4(cw.y, p4, true) << 4) & lim;
    g.fbits = (byte_mask4(cw.x, p4, false) | byte_mask4(cw.y, p4, false) << 4) & lim;
    int incl = __popc(g.bits);
    const int cnt = incl;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    g.r_first = rank_before(P, seg) + incl - cnt;
  } else {
    g.r_first = seg * SEG + 8 * lane;
    g.xb = P.x_lo + g.r_first;
    const int room = P.x_hi - g.xb;
    g.bits = room >= 8 ? 0xffu : (room > 0 ? (1u << room) - 1u : 0u);
    g.fbits = g.bits;
  }
  return g;
}

// Segments that hold the ranks [ra, rb) of the phase.
template <bool FILTER>
__device__ __forceinline__ void segment_range(const PhaseView& P, int ra, int rb, int* seg_a, int* seg_b) {
  if (FILTER) {
    // G[.][ph] is nondecreasing over the nsegs + 1 rows; last row = number of participants
    int a = 0, b = P.nsegs;               // largest seg with G[seg] <= ra
    while (a < b) { const int m = (a + b + 1) >> 1; if (rank_before(P, m) <= ra) a = m; else b = m - 1; }
    *seg_a = a;
    a = 0; b = P.nsegs;                   // smallest seg with G[seg] >= rb
    while (a < b) { const int m = (a + b) >> 1; if (rank_before(P, m) >= rb) b = m; else a = m + 1; }
    *seg_b = a;
  } else {
    *seg_a = ra / SEG;
    *seg_b = (rb + SEG - 1) / SEG;
  }
}

// Visits ranks [ra, rb), all of which start inside the tile whose origin is `trel` rounds after
// the phase's first round (trel may be slightly negative) and whose ring half is `buf`: adds the
// two events of every run.  Warps take segments in turn; nothing is written to global memory and
// no block-wide barrier is needed.
template <bool FILTER>
__device__ __forceinline__ void visit_runs(FShared& sh, const PhaseView& P, int ra, int rb, int trel, int buf,
                                           bool dense) {
  if (ra >= rb) return;
  u32* const dA = sh.dA;
  u32* const dB = sh.dB;
  const u32 tau = P.tau, k = P.k;
  const int warp = threadIdx.x >> 5;
  // 16-byte loads need aligned rows; without the filter a lane's first position is x_lo + 8*(...)
  const bool vec = ((reinterpret_cast<uintptr_t>(P.S) | reinterpret_cast<uintptr_t>(P.O)) & 15u) == 0 && (FILTER || (P.x_lo & 3) == 0);
  int seg_a, seg_b;
  segment_range<FILTER>(P, ra, rb, &seg_a, &seg_b);
  for (int seg = seg_a + warp; seg < seg_b; seg += WARPS) {
    // The prompt lengths of the lane's eight positions do not depend on which of them take part:
    // where all eight exist and the rows are 16-byte aligned they are requested first, as two
    // 16-byte loads, so that they travel together with the class bytes instead of after them.
    const int xb0 = (FILTER ? 0 : P.x_lo) + seg * SEG + 8 * static_cast<int>(lane_id());
    const bool vload = vec && xb0 + 8 <= P.n_src;
    uint4 a0 = make_uint4(0, 0, 0, 0), a1 = a0;
    if (vload) {
      a0 = __ldg(reinterpret_cast<const uint4*>(P.S + xb0));
      a1 = __ldg(reinterpret_cast<const uint4*>(P.S + xb0) + 1);
    }
    const LaneGroup g = lane_group<FILTER>(P, seg);
    // of this lane's participants, entries [skip, skip + take) have ranks inside [ra, rb)
    const int cnt = __popc(g.bits);
    const int skip = max(0, ra - g.r_first);
    const int take = min(cnt, rb - g.r_first) - skip;
    if (__ballot_sync(0xffffffffu, take > 0) == 0) continue;
    u32 s_[8], o_[8];
    // a killed run lasts tau rounds whatever its response length: only completing jobs load it
    const u32 need_o = take > 0 ? g.fbits : 0u;
    if (vload) {
      s_[0] = a0.x; s_[1] = a0.y; s_[2] = a0.z; s_[3] = a0.w; s_[4] = a1.x; s_[5] = a1.y; s_[6] = a1.z; s_[7] = a1.w;
      if (FILTER) {
#pragma unroll
        for (int j = 0; j < 8; ++j) o_[j] = (need_o >> j & 1u) ? static_cast<u32>(__ldg(P.O + g.xb + j)) : 0xffffffffu;
      } else {
        const uint4 b0 = take > 0 ? __ldg(reinterpret_cast<const uint4*>(P.O + g.xb)) : make_uint4(0, 0, 0, 0);
        const uint4 b1 = take > 0 ? __ldg(reinterpret_cast<const uint4*>(P.O + g.xb) + 1) : make_uint4(0, 0, 0, 0);
        o_[0] = b0.x; o_[1] = b0.y; o_[2] = b0.z; o_[3] = b0.w; o_[4] = b1.x; o_[5] = b1.y; o_[6] = b1.z; o_[7] = b1.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        s_[j] = 0; o_[j] = 0xffffffffu;
        if (take > 0 && (g.bits >> j & 1u)) s_[j] = static_cast<u32>(__ldg(P.S + g.xb + j));
        if (need_o >> j & 1u) o_[j] = static_cast<u32>(__ldg(P.O + g.xb + j));
      }
    }
    u32 q = 0, rem = 0;      // start offset of the current rank inside the phase and its remainder
    if (take > 0) {
      const u32 r0 = static_cast<u32>(g.r_first + skip);
      u64 dq_, dr_;
      divmod_u(static_cast<u64>(r0) * tau, k, &dq_, &dr_);
      q = static_cast<u32>(dq_);
      rem = static_cast<u32>(dr_);
    }
    // Dense phases (several runs start per round): the runs of a lane that start in the round of
    // its first run are summed in registers, then equal rounds - contiguous lanes, because
    // consecutive ranks start in nondecreasing rounds - are summed across the warp with a
    // segmented scan, and one lane per round issues the atomics.  Runs that hold their whole
    // slot end together (start + tau), so their end events are combined the same way.
    const bool dn = dense;
    int seg_key = 0x7fffffff;
    u32 seg_all = 0, seg_full = 0, seg_cnt = 0;
    int idx = 0;             // index among this lane's participants
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      int sidx = -1, eidx = -1;
      u32 c = 0;
      const bool part = (g.bits >> j & 1u) != 0;
      const bool on = part && idx >= skip && idx < skip + take;
      if (part) ++idx;
      if (on) {
        const u32 oi = o_[j];
        const u32 d = oi < tau ? oi : tau;
        c = s_[j] + 1u - P.base - q;                          // tokens(t) = c + t while active
        const int srel = static_cast<int>(q) - trel;
        sidx = ring(buf, srel);
        if (q + d < P.len) {                                   // an end at the phase end is never read
          const u32 erel = static_cast<u32>(srel) + d;
          if (erel < 2u * TILE) eidx = ring(buf, static_cast<int>(erel));
        }
        if (dn) {
          if (seg_key == 0x7fffffff) seg_key = srel;
          if (srel == seg_key) {
            seg_all += c; seg_cnt += 1u;
            sidx = -1;
            if (d == tau) { seg_full += c; seg_cnt += 1u << 16; eidx = -1; }
          }
        }
        rem += P.rt; q += P.qt;
        if (rem >= k) { rem -= k; ++q; }
      }
      if (sidx >= 0) { atomicAdd(&dA[sidx], c); atomicAdd(&dB[sidx], 1u); }
      if (eidx >= 0) { atomicAdd(&dA[eidx], 0u - c); atomicAdd(&dB[eidx], 0xffffffffu); }
    }
    if (dn) {
      // a lane without runs takes the round of the nearest lane before it that has some, so that
      // equal rounds stay contiguous for the segmented scan
      const u32 has = __ballot_sync(0xffffffffu, seg_key != 0x7fffffff);
      const u32 before = has & lanemask_lt();
      const int src = (seg_key == 0x7fffffff && before) ? 31 - __clz(before) : static_cast<int>(lane_id());
      int key = __shfl_sync(0xffffffffu, seg_key, src);
      u32 va = seg_all, vf = seg_full, vn = seg_cnt;
#pragma unroll
      for (int dd = 1; dd < 32; dd <<= 1) {
        const int kk = __shfl_up_sync(0xffffffffu, key, dd);
        const u32 ya = __shfl_up_sync(0xffffffffu, va, dd), yf = __shfl_up_sync(0xffffffffu, vf, dd);
        const u32 yn = __shfl_up_sync(0xffffffffu, vn, dd);
        if (static_cast<int>(lane_id()) >= dd && kk == key) { va += ya; vf += yf; vn += yn; }
      }
      const int next_key = __shfl_down_sync(0xffffffffu, key, 1);
      if (key != 0x7fffffff && (lane_id() == 31 || next_key != key)) {   // last lane of its round
        const int si = ring(buf, key);
        atomicAdd(&dA[si], va);
        atomicAdd(&dB[si], vn & 0xffffu);
        const u32 n_full = vn >> 16;
        // start offset of this round inside the phase: key + trel
        if (n_full && static_cast<u32>(key + trel) + tau < P.len) {
          const int ei = ring(buf, key + static_cast<int>(tau));          // tau < TILE in dense phases
          atomicAdd(&dA[ei], 0u - vf);
          atomicAdd(&dB[ei], 0u - n_full);
        }
      }
    }
  }
}

// The run visit where rank and position go together (exact keys: batching classes, SPS, simultaneous batches) and few runs
// start in a tile: one run per thread, so that a tile's runs are spread over the whole block.  (A warp that takes 256 positions,
// eight per lane, leaves the other warps idle: 6,500 cycles for a tile of 100 runs, 25,000 for one of 330 simultaneous runs.)
// Runs of one simultaneous batch start together: a warp of one batch books them with one atomic.
template <bool SIM>
__device__ __forceinline__ void visit_thin(FShared& sh, const PhaseView& P, int ra, int rb, int trel, int buf, u64 kinv) {
  u32* const dA = sh.dA;
  u32* const dB = sh.dB;
  for (int r0 = ra; r0 < rb; r0 += T) {
    const int r = r0 + static_cast<int>(threadIdx.x);
    const bool on = r < rb;
    if (!SIM && !on) continue;
    u32 si = 0, oi = 0, q = 0;
    if (on) {
      si = static_cast<u32>(__ldg(P.S + P.x_lo + r));
      oi = static_cast<u32>(__ldg(P.O + P.x_lo + r));
      q = SIM ? static_cast<u32>(r) / P.k * P.tau : slot_mul(static_cast<u32>(r), P.tau, P.k, kinv);
    }
    const u32 d = min(oi, P.tau), c = si + 1u - P.base - q;
    const int srel = static_cast<int>(q) - trel;
    if (SIM) {
      const u32 here = __ballot_sync(0xffffffffu, on);
      if (here == 0) continue;
      const int first = __shfl_sync(0xffffffffu, srel, 0);
      const bool same = __all_sync(0xffffffffu, !on || srel == first);
      if (same) {
        const u32 cs = __reduce_add_sync(0xffffffffu, on ? c : 0u);
        if (lane_id() == 0) { const int si_ = ring(buf, srel); atomicAdd(&dA[si_], cs); atomicAdd(&dB[si_], static_cast<u32>(__popc(here))); }
      } else if (on) {
        const int si_ = ring(buf, srel);
        atomicAdd(&dA[si_], c); atomicAdd(&dB[si_], 1u);
      }
      if (!on) continue;
    } else {
      const int si_ = ring(buf, srel);
      atomicAdd(&dA[si_], c); atomicAdd(&dB[si_], 1u);
    }
    if (q + d < P.len) {                                       // an end at the phase end is never read
      const u32 erel = static_cast<u32>(srel) + d;
      if (erel < 2u * TILE) { const int ei = ring(buf, static_cast<int>(erel)); atomicAdd(&dA[ei], 0u - c); atomicAdd(&dB[ei], 0xffffffffu); }
    }
  }
}

// The run visit of a phase with carried jobs in which at least eight runs start per round (and the
// slice is shorter than a tile).  A lane's up to eight participants then start in one round or in
// two consecutive ones, so the lane first treats all of them as killed at the end of their slot:
// one start event and one end event per round, from sums over its participants, without a loop
// over runs.  Afterwards each participant that completes before the end of its slot moves its own
// end event from start + tau to start + o.  Same events in total as visit_runs<false, true>.
__device__ __forceinline__ void visit_runs_sliced(FShared& sh, const PhaseView& P, int ra, int rb, int trel, int buf, u64 kinv) {
  if (ra >= rb) return;
  u32* const dA = sh.dA;
  u32* const dB = sh.dB;
  const u32 tau = P.tau, k = P.k;
  const int warp = threadIdx.x >> 5;
  const bool vec = (reinterpret_cast<uintptr_t>(P.S) & 15u) == 0;
  int seg_a, seg_b;
  segment_range<true>(P, ra, rb, &seg_a, &seg_b);
  for (int seg = seg_a + warp; seg < seg_b; seg += WARPS) {
    const int xb0 = seg * SEG + 8 * static_cast<int>(lane_id());
    const bool vload = vec && xb0 + 8 <= P.n_src;
    uint4 a0 = make_uint4(0, 0, 0, 0), a1 = a0;
    if (vload) {
      a0 = __ldg(reinterpret_cast<const uint4*>(P.S + xb0));
      a1 = __ldg(reinterpret_cast<const uint4*>(P.S + xb0) + 1);
    }
    const LaneGroup g = lane_group<true>(P, seg);
    const int cnt = __popc(g.bits);
    const int skip = max(0, ra - g.r_first);
    const int take = min(cnt, rb - g.r_first) - skip;
    if (__ballot_sync(0xffffffffu, take > 0) == 0) continue;
    if (take <= 0) continue;
    // the lane's participants with ranks inside [ra, rb)
    u32 bits = g.bits;
    for (int i = 0; i < skip; ++i) bits &= bits - 1u;
    for (int extra = __popc(bits) - take; extra > 0; --extra) bits &= ~(0x80000000u >> __clz(bits));
    u32 s_[8];
    if (vload) {
      s_[0] = a0.x; s_[1] = a0.y; s_[2] = a0.z; s_[3] = a0.w; s_[4] = a1.x; s_[5] = a1.y; s_[6] = a1.z; s_[7] = a1.w;
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) s_[j] = (bits >> j & 1u) ? static_cast<u32>(__ldg(P.S + g.xb + j)) : 0u;
    }
    const u32 n = static_cast<u32>(take);
    const u32 r0 = static_cast<u32>(g.r_first + skip);
    const u32 q0 = slot_mul(r0, tau, k, kinv);
    // rank r0 + j starts in round q0 + floor((rem + j tau) / k): the first m stay in round q0
    const u32 rem = static_cast<u32>(static_cast<u64>(r0) * tau - static_cast<u64>(q0) * k);
    u32 m = 1;
#pragma unroll
    for (u32 j = 1; j < 8; ++j) m += (rem + j * tau < k) ? 1u : 0u;
    m = min(m, n);
    u32 sumA = 0, sumB = 0, idx = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (bits >> j & 1u) {
        const u32 v = s_[j] + 1u;
        if (idx < m) sumA += v; else sumB += v;
        ++idx;
      }
    }
    const int srel = static_cast<int>(q0) - trel;
    {
      const u32 c = sumA - m * (P.base + q0);
      const int si = ring(buf, srel);
      atomicAdd(&dA[si], c);
      atomicAdd(&dB[si], m);
      if (q0 + tau < P.len) {
        const int ei = ring(buf, srel + static_cast<int>(tau));
        atomicAdd(&dA[ei], 0u - c);
        atomicAdd(&dB[ei], 0u - m);
      }
    }
    if (n > m) {
      const u32 c = sumB - (n - m) * (P.base + q0 + 1u);
      const int si = ring(buf, srel + 1);
      atomicAdd(&dA[si], c);
      atomicAdd(&dB[si], n - m);
      if (q0 + 1u + tau < P.len) {
        const int ei = ring(buf, srel + 1 + static_cast<int>(tau));
        atomicAdd(&dA[ei], 0u - c);
        atomicAdd(&dB[ei], 0u - (n - m));
      }
    }
    // completing jobs: the end moves from start + tau to start + o
    u32 fb = g.fbits & bits;
    while (fb) {
      const int j = __ffs(static_cast<int>(fb)) - 1;
      fb &= fb - 1u;
      const u32 oi = static_cast<u32>(__ldg(P.O + g.xb + j));
      if (oi < tau) {
        const u32 before = static_cast<u32>(__popc(bits & ((1u << j) - 1u)));
        const u32 q = q0 + (before >= m ? 1u : 0u);
        const u32 c = static_cast<u32>(__ldg(P.S + g.xb + j)) + 1u - P.base - q;
        const int sr = static_cast<int>(q) - trel;
        if (q + oi < P.len) {
          const int ei = ring(buf, sr + static_cast<int>(oi));
          atomicAdd(&dA[ei], 0u - c);
          atomicAdd(&dB[ei], 0xffffffffu);
        }
        if (q + tau < P.len) {
          const int ki = ring(buf, sr + static_cast<int>(tau));
          atomicAdd(&dA[ki], c);
          atomicAdd(&dB[ki], 1u);
        }
      }
    }
  }
}

// Exclusive block scan of a small per-thread count; returns this thread's offset, total in *total.
__device__ __forceinline__ int block_count_scan(int v, int* red32, int* total) {
  int incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, d);
    if (static_cast<int>(lane_id()) >= d) incl += y;
  }
  const int warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane_id() == 31) red32[warp] = incl;
  __syncthreads();
  const int w = (lane_id() < WARPS) ? red32[lane_id()] : 0;
  int wi = w;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, wi, d);
    if (static_cast<int>(lane_id()) >= d) wi += y;
  }
  *total = __shfl_sync(0xffffffffu, wi, 31);
  return __shfl_sync(0xffffffffu, wi - w, warp) + (incl - v);
}

// Participants of a phase as a list (used once fewer than half of a window's positions still take
// part): rank r < C is the (s, o) pair cur[r], rank r >= C is position src + (r - C) of the
// window (jobs that enter in this phase).
struct ListView {
  const uint2* cur;
  int C;
  int src;
  int cap;                // entries of either list in this CTA's scratch
};

// Run visit over a list: ranks [ra, rb), one to four consecutive ranks per thread, so that a tile
// with few runs is spread over the whole block instead of a few warps.  Adds the two events of
// every run and appends the killed jobs to `nxt`; returns the new length of `nxt`.  Block-wide
// (two barriers per 2048 ranks for the positions of the survivors).
__device__ __forceinline__ int visit_list(FShared& sh, const PhaseView& P, const ListView& V, uint2* nxt, int C_next,
                                          int ra, int rb, int trel, int buf, bool dense) {
  const int tid = threadIdx.x, lane = lane_id();
  u32* const dA = sh.dA;
  u32* const dB = sh.dB;
  const u32 tau = P.tau, k = P.k;
  for (int c0 = ra; c0 < rb;) {
    const int left = rb - c0;
    const int rpt = left > 2 * T ? RPT : (left > T ? 2 : 1);
    const int r_first = c0 + tid * rpt;
    c0 += T * rpt;
    uint2 keep[RPT];
    u32 cmask = 0;
    if (r_first - lane * rpt < rb) {   // warps past the end of the range skip the visit
      u32 s_[RPT], o_[RPT];
      bool on[RPT];
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const int r = r_first + j;
        on[j] = j < rpt && r < rb;
        s_[j] = 0; o_[j] = 0;
        if (on[j]) {
          if (r < V.C) { if (KVS_IN(r, V.cap, CHK_LIST)) { const uint2 e = V.cur[r]; s_[j] = e.x; o_[j] = e.y; } }
          else { s_[j] = static_cast<u32>(__ldg(P.S + V.src + (r - V.C))); o_[j] = static_cast<u32>(__ldg(P.O + V.src + (r - V.C))); }
        }
      }
      u32 q = 0, rem = 0;
      if (on[0]) {
        u64 dq_, dr_;
        divmod_u(static_cast<u64>(r_first) * tau, k, &dq_, &dr_);
        q = static_cast<u32>(dq_);
        rem = static_cast<u32>(dr_);
      }
      int seg_key = 0x7fffffff;
      u32 seg_all = 0, seg_full = 0, seg_cnt = 0;
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        if (on[j]) {
          const u32 oi = o_[j];
          const u32 d = oi < tau ? oi : tau;
          if (oi > tau) { keep[j] = make_uint2(s_[j], oi); cmask |= 1u << j; }
          const u32 c = s_[j] + 1u - P.base - q;
          const int srel = static_cast<int>(q) - trel;
          int sidx = ring(buf, srel), eidx = -1;
          if (q + d < P.len) {
            const u32 erel = static_cast<u32>(srel) + d;
            if (erel < 2u * TILE) eidx = ring(buf, static_cast<int>(erel));
          }
          if (dense) {
            if (seg_key == 0x7fffffff) seg_key = srel;
            if (srel == seg_key) {
              seg_all += c; seg_cnt += 1u;
              sidx = -1;
              if (d == tau) { seg_full += c; seg_cnt += 1u << 16; eidx = -1; }
            }
          }
          if (sidx >= 0) { atomicAdd(&dA[sidx], c); atomicAdd(&dB[sidx], 1u); }
          if (eidx >= 0) { atomicAdd(&dA[eidx], 0u - c); atomicAdd(&dB[eidx], 0xffffffffu); }
          rem += P.rt; q += P.qt;
          if (rem >= k) { rem -= k; ++q; }
        }
      }
      if (dense) {
        const u32 has = __ballot_sync(0xffffffffu, seg_key != 0x7fffffff);
        const u32 before = has & lanemask_lt();
        const int src = (seg_key == 0x7fffffff && before) ? 31 - __clz(before) : lane;
        const int key = __shfl_sync(0xffffffffu, seg_key, src);
        u32 va = seg_all, vf = seg_full, vn = seg_cnt;
#pragma unroll
        for (int dd = 1; dd < 32; dd <<= 1) {
          const int kk = __shfl_up_sync(0xffffffffu, key, dd);
          const u32 ya = __shfl_up_sync(0xffffffffu, va, dd), yf = __shfl_up_sync(0xffffffffu, vf, dd);
          const u32 yn = __shfl_up_sync(0xffffffffu, vn, dd);
          if (lane >= dd && kk == key) { va += ya; vf += yf; vn += yn; }
        }
        const int next_key = __shfl_down_sync(0xffffffffu, key, 1);
        if (key != 0x7fffffff && (lane == 31 || next_key != key)) {
          const int si = ring(buf, key);
          atomicAdd(&dA[si], va);
          atomicAdd(&dB[si], vn & 0xffffu);
          const u32 n_full = vn >> 16;
          if (n_full && static_cast<u32>(key + trel) + tau < P.len) {
            const int ei = ring(buf, key + static_cast<int>(tau));
            atomicAdd(&dA[ei], 0u - vf);
            atomicAdd(&dB[ei], 0u - n_full);
          }
        }
      }
    }
    int total;
    int off = C_next + block_count_scan(__popc(cmask), sh.red32, &total);
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (cmask >> j & 1u) { if (KVS_IN(off, V.cap, CHK_LIST_OUT)) nxt[off] = keep[j]; ++off; }
    C_next += total;
  }
  return C_next;
}

// insert_far_ends for a list: slices longer than a tile only.
__device__ __forceinline__ void insert_far_ends_list(FShared& sh, const PhaseView& P, const ListView& V, int N, int a0,
                                                     int u0, int wlen, int buf) {
  if (u0 <= TILE) return;
  const u32 lo = static_cast<u32>(u0) > P.tau ? static_cast<u32>(u0) - P.tau : 0u, hi = static_cast<u32>(u0 - TILE);
  i64 r_lo = ceil_div_u(static_cast<u64>(lo) * P.k, P.tau), r_hi = ceil_div_u(static_cast<u64>(hi) * P.k, P.tau);
  if (r_hi > N) r_hi = N;
  for (i64 r0 = r_lo; r0 < r_hi; r0 += T) {
    const i64 rr = r0 + threadIdx.x;
    if (rr < r_hi) {
      const int r = static_cast<int>(rr);
      u32 si, oi;
      if (r < V.C) { uint2 e = make_uint2(0, 1); if (KVS_IN(r, V.cap, CHK_LIST)) e = V.cur[r]; si = e.x; oi = e.y; }
      else { si = static_cast<u32>(__ldg(P.S + V.src + (r - V.C))); oi = static_cast<u32>(__ldg(P.O + V.src + (r - V.C))); }
      const u32 q = slot32(static_cast<u32>(r), P.tau, P.k);
      const u32 end = q + (oi < P.tau ? oi : P.tau);
      const int ts = a0 + ((static_cast<int>(q) - a0) / TILE) * TILE;
      if (static_cast<int>(end) >= ts + 2 * TILE && static_cast<int>(end) >= u0 && static_cast<int>(end) < u0 + wlen && end < P.len) {
        const u32 c = si + 1u - P.base - q;
        const int ei = ring(buf, static_cast<int>(end) - u0);
        atomicAdd(&sh.dA[ei], 0u - c);
        atomicAdd(&sh.dB[ei], 0xffffffffu);
      }
    }
  }
}

// A phase in which every position of the window takes part and none completes (index order, all
// response lengths beyond the slice: the early phases of the slicing algorithm) needs no visit of
// its runs.  Rank = position, every run lasts tau rounds, so the events of a round are sums over
// position ranges: with PS[x] = sum of (s + 1) over positions below x and B(u) = number of ranks that
// start in round u or earlier = min(N, ceil((u + 1) k / tau)), the runs that start in round u add
// (PS[B(u)] - PS[B(u-1)] - cnt (base + u), cnt) there and the opposite tau rounds later.  Each thread
// forms the events of its own ITEMS rounds of the tile - starts at u and ends of the runs started
// at u - tau - and adds them to its own words of the ring: no atomics, no dependence on the number
// of runs.  u0 = offset of the tile's origin inside the phase.
__device__ __forceinline__ void pure_phase_events(FShared& sh, const PhaseView& P, const u32* __restrict__ PS, int ps_cap, int N, int u0, int buf) {
  (void)ps_cap;
  const int e0 = ITEMS * static_cast<int>(threadIdx.x);
  const int w0 = ring(buf, e0);
  const u32 tau = P.tau, k = P.k;
  const u32 kq = k / tau, kr = k - kq * tau;          // k = kq * tau + kr
#pragma unroll
  for (int stream = 0; stream < 2; ++stream) {
    // stream 0: runs that start in the thread's rounds; stream 1: runs that end there (started tau earlier)
    const i64 ufirst = static_cast<i64>(u0) + e0 - (stream ? static_cast<i64>(tau) : 0);   // start round of the first event
    // B(ufirst - 1) by one division, then stepped: (u + 1) k = Q tau + R
    u64 Q = 0, R = 0;
    i64 u = ufirst - 1;
    if (u >= 0) divmod_u(static_cast<u64>(u + 1) * k, tau, &Q, &R);
    u32 b_prev = u >= 0 ? static_cast<u32>(min(static_cast<u64>(N), Q + (R > 0))) : 0u;
    u32 ps_prev = KVS_IN(b_prev, ps_cap, CHK_PS) ? PS[b_prev] : 0u;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      ++u;
      if (u == 0) { Q = kq; R = kr; }                  // (0 + 1) k
      else if (u > 0) { Q += kq; R += kr; if (R >= tau) { R -= tau; ++Q; } }
      const i64 land = u + (stream ? static_cast<i64>(tau) : 0);          // round the event lands in
      if (u >= 0 && land < static_cast<i64>(P.len)) {
        const u32 b = static_cast<u32>(min(static_cast<u64>(N), Q + (R > 0)));
        if (b != b_prev) {
          const u32 ps = KVS_IN(b, ps_cap, CHK_PS) ? PS[b] : 0u;
          const u32 cnt = b - b_prev;
          const u32 c = (ps - ps_prev) - cnt * (P.base + static_cast<u32>(u));
          if (stream == 0) { sh.dA[w0 + i] += c; sh.dB[w0 + i] += cnt; }
          else { sh.dA[w0 + i] -= c; sh.dB[w0 + i] -= cnt; }
          b_prev = b; ps_prev = ps;
        }
      }
    }
  }
}

// Slices longer than a tile: ends that land two or more tiles after the run's start were not
// inserted when the run was visited; pick them up when their tile comes.  u0 = offset of this
// tile's origin inside the phase, a0 = the same for the phase's first tile (0 or slightly negative).
template <bool FILTER>
__device__ __forceinline__ void insert_far_ends(FShared& sh, const PhaseView& P, bool sim, int N, int a0, int u0,
                                                int wlen, int buf) {
  if (u0 <= TILE) return;
  const u32 lo = static_cast<u32>(u0) > P.tau ? static_cast<u32>(u0) - P.tau : 0u, hi = static_cast<u32>(u0 - TILE);
  i64 r_lo, r_hi;   // ranks whose start offset lies in [lo, hi)
  if (sim) { r_lo = ceil_div_u(lo, P.tau) * P.k; r_hi = ceil_div_u(hi, P.tau) * P.k; }
  else { r_lo = ceil_div_u(static_cast<u64>(lo) * P.k, P.tau); r_hi = ceil_div_u(static_cast<u64>(hi) * P.k, P.tau); }
  if (r_hi > N) r_hi = N;
  if (r_lo >= r_hi) return;
  const int ra = static_cast<int>(r_lo), rb = static_cast<int>(r_hi);
  u32* const dA = sh.dA;
  u32* const dB = sh.dB;
  const int warp = threadIdx.x >> 5;
  int seg_a, seg_b;
  segment_range<FILTER>(P, ra, rb, &seg_a, &seg_b);
  for (int seg = seg_a + warp; seg < seg_b; seg += WARPS) {
    const LaneGroup g = lane_group<FILTER>(P, seg);
    int r = g.r_first;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (!(g.bits >> j & 1u)) continue;
      const int rr = r++;
      if (rr < ra || rr >= rb) continue;
      const u32 si = static_cast<u32>(__ldg(P.S + g.xb + j)), oi = static_cast<u32>(__ldg(P.O + g.xb + j));
      const u32 q = sim ? (static_cast<u32>(rr) / P.k) * P.tau : slot32(static_cast<u32>(rr), P.tau, P.k);
      const u32 end = q + (oi < P.tau ? oi : P.tau);
      const int ts = a0 + ((static_cast<int>(q) - a0) / TILE) * TILE;   // origin of the tile the run started in
      if (static_cast<int>(end) >= ts + 2 * TILE && static_cast<int>(end) >= u0 && static_cast<int>(end) < u0 + wlen && end < P.len) {
        const u32 c = si + 1u - P.base - q;
        const int ei = ring(buf, static_cast<int>(end) - u0);
        atomicAdd(&dA[ei], 0u - c);
        atomicAdd(&dB[ei], 0xffffffffu);
      }
    }
  }
}

// A phase whose rounds are walked from a tile in its middle on (u0 = offset of that tile inside the phase): what the runs
// that started before hold in round u0 (sums over the threads), and the ends in this tile of those that started in
// the tile before (ends of earlier ones are picked up by insert_far_ends).
struct CarryIn { u32 A, B; };
__device__ __forceinline__ void carry_in_run(FShared& sh, const PhaseView& P, CarryIn& c, u32 si, u32 oi, u32 q, int u0, int buf) {
  const u32 end = q + min(oi, P.tau);
  if (end < static_cast<u32>(u0)) return;
  const u32 v = si + 1u - P.base - q;
  c.A += v;
  c.B += 1u;
  if (static_cast<int>(q) >= u0 - TILE && end < static_cast<u32>(u0 + TILE) && end < P.len) {
    const int ei = ring(buf, static_cast<int>(end) - u0);
    atomicAdd(&sh.dA[ei], 0u - v);
    atomicAdd(&sh.dB[ei], 0xffffffffu);
  }
}
template <bool FILTER>
__device__ __forceinline__ CarryIn carry_in(FShared& sh, const PhaseView& P, bool sim, int ra, int rb, int u0, int buf) {
  CarryIn c{0, 0};
  if (ra >= rb) return c;
  int seg_a, seg_b;
  segment_range<FILTER>(P, ra, rb, &seg_a, &seg_b);
  for (int seg = seg_a + static_cast<int>(threadIdx.x >> 5); seg < seg_b; seg += WARPS) {
    const LaneGroup g = lane_group<FILTER>(P, seg);
    int r = g.r_first;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (!(g.bits >> j & 1u)) continue;
      const int rr = r++;
      if (rr < ra || rr >= rb) continue;
      const u32 q = sim ? (static_cast<u32>(rr) / P.k) * P.tau : slot32(static_cast<u32>(rr), P.tau, P.k);
      carry_in_run(sh, P, c, static_cast<u32>(__ldg(P.S + g.xb + j)), static_cast<u32>(__ldg(P.O + g.xb + j)), q, u0, buf);
    }
  }
  return c;
}
__device__ __forceinline__ CarryIn carry_in_list(FShared& sh, const PhaseView& P, const ListView& V, int ra, int rb, int u0, int buf) {
  CarryIn c{0, 0};
  for (int r = ra + static_cast<int>(threadIdx.x); r < rb; r += T) {
    uint2 e = make_uint2(0, 1);
    if (r < V.C) { if (KVS_IN(r, V.cap, CHK_LIST)) e = V.cur[r]; }
    else e = make_uint2(static_cast<u32>(__ldg(P.S + V.src + (r - V.C))), static_cast<u32>(__ldg(P.O + V.src + (r - V.C))));
    carry_in_run(sh, P, c, e.x, e.y, slot32(static_cast<u32>(r), P.tau, P.k), u0, buf);
  }
  return c;
}
// The same where every position takes part and none completes: closed forms, in every thread.
__device__ __forceinline__ CarryIn carry_in_pure(const PhaseView& P, const u32* __restrict__ PS, int N, int u0) {
  auto started = [&](i64 u) -> u64 {            // ranks that start in round u or earlier
    if (u < 0) return 0;
    const u64 b = static_cast<u64>(ceil_div_u(static_cast<u64>(u + 1) * P.k, P.tau));
    return b < static_cast<u64>(N) ? b : static_cast<u64>(N);
  };
  const u64 a = started(static_cast<i64>(u0) - 1 - P.tau), b = started(static_cast<i64>(u0) - 1);
  const u32 cnt = static_cast<u32>(b - a);
  const u32 starts = static_cast<u32>(floor_sum(b, P.k, P.tau, 0) - floor_sum(a, P.k, P.tau, 0));
  return CarryIn{PS[b] - PS[a] - cnt * P.base - starts, cnt};
}

// Exclusive prefix sums (modulo 2^32) of f(0) .. f(n - 1) over the block: out[0 .. n].
template <class F>
__device__ __forceinline__ void block_prefix(FShared& sh, u32* out, int out_cap, int n, F f) {
  const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  (void)out_cap;
  u32 run = 0;
  for (int x0 = 0; x0 <= n; x0 += T * 4) {
    const int x = x0 + 4 * tid;
    u32 in[4], v[4], tot = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) in[j] = x + j < n ? f(x + j) : 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) { v[j] = tot; tot += in[j]; }
    const u32 incl = warp_incl(tot);
    __syncthreads();
    if (lane == 31) sh.redA[warp] = incl;
    __syncthreads();
    const u32 w = lane < WARPS ? sh.redA[lane] : 0u;
    const u32 wi = warp_incl(w);
    const u32 off = run + __shfl_sync(0xffffffffu, wi - w, warp) + (incl - tot);
    run += __shfl_sync(0xffffffffu, wi, 31);
#pragma unroll
    for (int j = 0; j < 4; ++j) if (x + j <= n && KVS_IN(x + j, out_cap, CHK_PS)) out[x + j] = off + v[j];
  }
  __syncthreads();
}

// Peak of one staggered phase without its rounds: memory grows between the ends of runs, so its maximum is the memory in
// the last round of some run, summed here over the ranks that have started and whose slots have not ended then - at
// most k of them.  job(r) = (s, o) of rank r.  First every rank's s less its start and its end go to `list` (which may be where
// job reads from), so that a pair of a run end and a rank costs a load, a comparison and two additions.  Of the run ends this CTA
// takes those of `part` of `parts`.  Returns this thread's maximum.
template <class F>
__device__ __forceinline__ u32 ends_peak(uint2* list, int list_cap, u32 N, u32 tau, u32 k, u64 kinv, int part, int parts, F job) {
  (void)list_cap;
  for (u32 r = threadIdx.x; r < N; r += T) {
    const uint2 e = job(static_cast<int>(r));
    const u32 q = slot_mul(r, tau, k, kinv);
    if (KVS_IN(r, list_cap, CHK_LIST_OUT)) list[r] = make_uint2(e.x - q, q + min(e.y, tau));
  }
  __syncthreads();
  u32 peak = 0;
  for (u32 i = threadIdx.x + static_cast<u32>(part) * T; i < N; i += static_cast<u32>(parts) * T) {
    const u32 t1 = list[i].y;                                      // last round of the run, plus one
    const u32 rb = static_cast<u32>(min_i64(N, ceil_div_u(static_cast<u64>(t1) * k, tau)));
    const u32 ra = t1 <= tau ? 0u : static_cast<u32>(ceil_div_u(static_cast<u64>(t1 - tau) * k, tau));
    u32 sum = 0, cnt = 0;
#pragma unroll 4
    for (u32 r = ra; r < rb; ++r) {
      const uint2 e = list[r];
      if (e.y >= t1) { sum += e.x; ++cnt; }
    }
    peak = max(peak, sum + cnt * t1);
  }
  return peak;
}

// end of the batch of k ranks that holds rank r, of N
__device__ __forceinline__ u32 batch_end(u32 r, u32 k, u32 N) {
  return static_cast<u32>(min(static_cast<u64>(N), static_cast<u64>(r / k + 1) * k));
}

// Largest batch of kk ranks: its difference of the prefix sums PS plus d for each of its jobs.  Returns this thread's maximum.
__device__ __forceinline__ u32 widest_batch(const u32* PS, int ps_cap, u32 N, u32 kk, u32 d) {
  (void)ps_cap;
  u32 W = 0;
  for (u64 i = static_cast<u64>(threadIdx.x) * kk; i < N; i += static_cast<u64>(T) * kk) {
    const u32 a = static_cast<u32>(i), b = static_cast<u32>(min(static_cast<u64>(N), static_cast<u64>(i + kk)));
    if (KVS_IN(b, ps_cap, CHK_PS)) W = max(W, PS[b] - PS[a] + (b - a) * d);
  }
  return W;
}

// Peak of one phase that runs in batches of kk ranks: the jobs of a batch start together and end after d in (low, tau]
// rounds, so memory after d rounds is the sum of s + d over those that last for d or longer.  Short slices hold large
// batches: one bucket per batch and d, as many as there are rounds in which a run can end, summed tile by tile; long slices
// hold small ones: one pass over its batch for every job.  Cycles of a CTA, roughly: 3,000 per tile against 24 per job
// and step of the block.  PS: prefix sums of s over the ranks.  Returns this thread's maximum.
__device__ __forceinline__ u32 batches_peak(FShared& sh, const uint2* list, const u32* PS, int list_cap, u32 N, u32 kk, u32 tau, u32 low) {
  (void)list_cap;
  const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  const u32 W = tau - low;
  const u64 n_v = static_cast<u64>((N + kk - 1) / kk) * W;         // buckets, below the rounds of the phase
  const u64 n_tiles = (n_v + TILE - 1) / TILE;
  const u64 by_pairs = static_cast<u64>((N + T - 1) / T) * kk * 24;
  u32 peak = 0;
  if (by_pairs <= n_tiles * 3000) {
    for (u32 i = tid; i < N; i += T) {
      const u32 b0 = (i / kk) * kk, b1 = min(N, b0 + kk);
      const u32 d = min(KVS_IN(i, list_cap, CHK_LIST) ? list[i].y : 1u, tau);
      u32 sum = 0, cnt = 0;
#pragma unroll 4
      for (u32 r = b0; r < b1; ++r) {
        const uint2 e = list[r];
        if (e.y >= d) { sum += e.x; ++cnt; }
      }
      peak = max(peak, sum + cnt * d);
    }
    return peak;
  }
  u32 A = 0, B = 0;                                                // sum of s and number of the jobs in earlier tiles
  for (u32 v0 = 0; v0 < n_v; v0 += TILE) {
    const u32 first = (v0 / W) * kk;
    const u32 last = static_cast<u32>(min(static_cast<u64>(N), (static_cast<u64>((v0 + TILE - 1) / W) + 1) * kk));
    for (u32 r = first + tid; r < last; r += T) {
      const uint2 e = KVS_IN(r, list_cap, CHK_LIST) ? list[r] : make_uint2(0, 1);
      const u32 x = (r / kk) * W + (min(e.y, tau) - 1u - low) - v0;
      if (x < static_cast<u32>(TILE)) { atomicAdd(&sh.dA[ring(0, static_cast<int>(x))], e.x); atomicAdd(&sh.dB[ring(0, static_cast<int>(x))], 1u); }
    }
    __syncthreads();
    const int w0 = ring(0, ITEMS * tid);
    u32 a[ITEMS], b[ITEMS], sa = 0, sb = 0;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {                              // exclusive sums
      a[i] = sa; b[i] = sb;
      sa += sh.dA[w0 + i]; sb += sh.dB[w0 + i];
      sh.dA[w0 + i] = 0; sh.dB[w0 + i] = 0;
    }
    u32 ia = sa, ib = sb;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 ya = __shfl_up_sync(0xffffffffu, ia, d), yb = __shfl_up_sync(0xffffffffu, ib, d);
      if (lane >= d) { ia += ya; ib += yb; }
    }
    if (lane == 31) { sh.redA[warp] = ia; sh.redB[warp] = ib; }
    __syncthreads();
    u32 wa = lane < WARPS ? sh.redA[lane] : 0u, wb = lane < WARPS ? sh.redB[lane] : 0u;
    const u32 wa0 = wa, wb0 = wb;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const u32 ya = __shfl_up_sync(0xffffffffu, wa, d), yb = __shfl_up_sync(0xffffffffu, wb, d);
      if (lane >= d) { wa += ya; wb += yb; }
    }
    const u32 offA = A + __shfl_sync(0xffffffffu, wa - wa0, warp) + (ia - sa);
    const u32 offB = B + __shfl_sync(0xffffffffu, wb - wb0, warp) + (ib - sb);
    A += __shfl_sync(0xffffffffu, wa, 31);
    B += __shfl_sync(0xffffffffu, wb, 31);
    u32 v = v0 + ITEMS * tid, bt = v / W, x = v - bt * W;
    u32 bend = batch_end(bt * kk, kk, N), ps = v < n_v ? PS[bend] : 0u;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i, ++v, ++x) {
      if (x == W) {
        x = 0; ++bt;
        if (v < n_v) { bend = batch_end(bt * kk, kk, N); ps = PS[bend]; }
      }
      // those that have not ended in an earlier bucket, in round low + x + 1 of their slot
      if (v < n_v) peak = max(peak, ps - (offA + a[i]) + (bend - (offB + b[i])) * (low + x + 1u));
    }
    __syncthreads();
  }
  return peak;
}

// Participants of a carried phase as a list in rank order.  All loads of a segment are issued before the first store.
__device__ __forceinline__ void list_participants(const PhaseView& P, uint2* list, int list_cap) {
  (void)list_cap;
  const bool vec = ((reinterpret_cast<uintptr_t>(P.S) | reinterpret_cast<uintptr_t>(P.O)) & 15u) == 0;
  for (int seg = threadIdx.x >> 5; seg < P.nsegs; seg += WARPS) {
    const int xb = seg * SEG + 8 * static_cast<int>(lane_id());
    u32 s_[8], o_[8];
    if (vec && xb + 8 <= P.n_src) {
      const uint4 a0 = __ldg(reinterpret_cast<const uint4*>(P.S + xb)), a1 = __ldg(reinterpret_cast<const uint4*>(P.S + xb) + 1);
      const uint4 b0 = __ldg(reinterpret_cast<const uint4*>(P.O + xb)), b1 = __ldg(reinterpret_cast<const uint4*>(P.O + xb) + 1);
      s_[0] = a0.x; s_[1] = a0.y; s_[2] = a0.z; s_[3] = a0.w; s_[4] = a1.x; s_[5] = a1.y; s_[6] = a1.z; s_[7] = a1.w;
      o_[0] = b0.x; o_[1] = b0.y; o_[2] = b0.z; o_[3] = b0.w; o_[4] = b1.x; o_[5] = b1.y; o_[6] = b1.z; o_[7] = b1.w;
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int x = min(xb + j, P.n_src - 1);          // past the end: a job that does not take part
        s_[j] = static_cast<u32>(__ldg(P.S + x));
        o_[j] = static_cast<u32>(__ldg(P.O + x));
      }
    }
    const LaneGroup g = lane_group<true>(P, seg);
    int r = g.r_first;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (g.bits >> j & 1u) {
        if (KVS_IN(r, list_cap, CHK_LIST_OUT)) list[r] = make_uint2(s_[j], o_[j]);
        ++r;
      }
  }
  __syncthreads();
}

// Prefix-sums one tile of the ring, turns it into memory(t), reduces the peak, stores the profile
// and leaves the tile zeroed for its next use.  Contains one __syncthreads.  t0 = absolute round
// of the tile's origin; rounds [first_round, t0 + wlen) below prof_cap are stored.
__device__ __forceinline__ void scan_tile(FShared& sh, int buf, i64 t0, int wlen, u32 first_round,
                                          u32& A_run, u32& B_run, u32& peak, int32_t* prof, i64 prof_cap) {
  const int tid = threadIdx.x;
  const uint4 zero = make_uint4(0, 0, 0, 0);
  u32 a[ITEMS], b[ITEMS];
  const int w0 = ring(buf, ITEMS * tid);       // the thread's ITEMS rounds are consecutive words
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    uint4* const pa = reinterpret_cast<uint4*>(&sh.dA[w0 + 4 * v]);
    uint4* const pb = reinterpret_cast<uint4*>(&sh.dB[w0 + 4 * v]);
    const uint4 x = *pa, y = *pb;
    *pa = zero;
    *pb = zero;
    a[4 * v] = x.x; a[4 * v + 1] = x.y; a[4 * v + 2] = x.z; a[4 * v + 3] = x.w;
    b[4 * v] = y.x; b[4 * v + 1] = y.y; b[4 * v + 2] = y.z; b[4 * v + 3] = y.w;
  }
#pragma unroll
  for (int i = 1; i < ITEMS; ++i) { a[i] += a[i - 1]; b[i] += b[i - 1]; }
  const u32 sa = a[ITEMS - 1], sb = b[ITEMS - 1];
  u32 ia = sa, ib = sb;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const u32 ya = __shfl_up_sync(0xffffffffu, ia, d), yb = __shfl_up_sync(0xffffffffu, ib, d);
    if (static_cast<int>(lane_id()) >= d) { ia += ya; ib += yb; }
  }
  if (lane_id() == 31) { sh.redA[tid >> 5] = ia; sh.redB[tid >> 5] = ib; }
  __syncthreads();
  const u32 wa = (lane_id() < WARPS) ? sh.redA[lane_id()] : 0, wb = (lane_id() < WARPS) ? sh.redB[lane_id()] : 0;
  u32 wia = wa, wib = wb;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const u32 ya = __shfl_up_sync(0xffffffffu, wia, d), yb = __shfl_up_sync(0xffffffffu, wib, d);
    if (static_cast<int>(lane_id()) >= d) { wia += ya; wib += yb; }
  }
  const u32 offA = A_run + __shfl_sync(0xffffffffu, wia - wa, tid >> 5) + (ia - sa);
  const u32 offB = B_run + __shfl_sync(0xffffffffu, wib - wb, tid >> 5) + (ib - sb);
  A_run += __shfl_sync(0xffffffffu, wia, 31);
  B_run += __shfl_sync(0xffffffffu, wib, 31);
  const int e0 = tid * ITEMS;
  const u32 tt = static_cast<u32>(t0) + static_cast<u32>(e0);
  u32 mem[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) mem[i] = (offA + a[i]) + (tt + i) * (offB + b[i]);
  // a tile that lies inside the phase and inside the caller's capacity needs no per-round tests
  const bool whole = wlen == TILE && (prof_cap <= 0 || (t0 >= static_cast<i64>(first_round) && t0 + TILE <= prof_cap));
  if (whole) {
    u32 m = mem[0];
#pragma unroll
    for (int i = 1; i < ITEMS; ++i) m = max(m, mem[i]);
    peak = max(peak, m);
    if (prof_cap > 0 && KVS_IN(t0 + e0, prof_cap - (ITEMS - 1), CHK_PROFILE)) {
      int4* dst = reinterpret_cast<int4*>(prof + t0 + e0);
#pragma unroll
      for (int v = 0; v < VEC; ++v)
        __stcs(&dst[v], make_int4(static_cast<int>(mem[4 * v]), static_cast<int>(mem[4 * v + 1]),
                                  static_cast<int>(mem[4 * v + 2]), static_cast<int>(mem[4 * v + 3])));   // written once, never re-read: streaming
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < ITEMS; ++i)
    if (e0 + i < wlen) peak = max(peak, mem[i]);
  if (prof_cap > 0) {
    const i64 lo = first_round, hi = min_i64(t0 + wlen, prof_cap);
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      const i64 rs = t0 + e0 + 4 * v;
      int32_t* dst = prof + rs;
      if (rs >= lo && rs + 4 <= hi && KVS_IN(rs, prof_cap - 3, CHK_PROFILE)) {
        *reinterpret_cast<int4*>(dst) = make_int4(static_cast<int>(mem[4 * v]), static_cast<int>(mem[4 * v + 1]),
                                                  static_cast<int>(mem[4 * v + 2]), static_cast<int>(mem[4 * v + 3]));
      } else if (rs + 4 > lo && rs < hi) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (rs + i >= lo && rs + i < hi && KVS_IN(rs + i, prof_cap, CHK_PROFILE)) dst[i] = static_cast<int>(mem[4 * v + i]);
      }
    }
  }
}

struct FAcc {
  u64 flow = 0, steps = 0;
  u32 hmax = 0;
  int unfinished = 0;
  u32 peak = 0;
};

// LIGHT: the variant for evaluations that walk no rounds (schedule only, or SPS / SimS whose peak
// comes from the run ends): no ring in shared memory and fewer registers, so that three CTAs fit an
// SM; an evaluation that needs its rounds walked is passed on to the full variant through a list.
// FAM: KVS_FUSED_ANY takes any evaluation, KVS_FUSED_SHARED (full variant) too and shares each between CTAs (in one kernel with the
// other, calls with estimates lost a tenth to spills); a family id (KVS_GBA .. KVS_SIMS) gives the kernel compiled
// for that family on exact response lengths only (the caller lists nothing else for it), so that
// each keeps just its own paths and gets its own register allocation.
// VARIANTS: with the code for simultaneous batches and per-phase prompt lengths.  The full batching kernel never has it (the light one
// takes those, or leaves them to the general kernel): 176 bytes of spills a thread with it, 12 without, 4,096 evaluations of 50,000
// jobs with their profiles 4.03 and 3.36 ms.  The kernel for shared evaluations exists with it, without it, and without it for calls
// with estimates (spill loads a thread 3,080, 2,328 and 1,840 bytes; one kernel for all three: 3,568): 64 instances of 50,000 jobs
// in windows 1,432 -> 1,270 us, four evaluations of 1,000 jobs 177 -> 170, 64 initial slices 429 -> 406.  The slicing
// kernel spills no less without it.
template <bool LIGHT, int FAM, bool VARIANTS>
__global__ void __launch_bounds__(KVS_EVAL_THREADS, LIGHT ? KVS_EVAL_MIN_CTAS + 1 : KVS_EVAL_MIN_CTAS) k_fused_eval(BuildParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FShared& sh = *reinterpret_cast<FShared*>(smem_raw);
  const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  // per-CTA scratch: class bytes of the current window (padded to whole segments), then the rank table
  unsigned char* const cls = reinterpret_cast<unsigned char*>(p.lists) + static_cast<i64>(blockIdx.x) * KVS_CTA_SCRATCH(p.max_jobs);
  u32* const G = reinterpret_cast<u32*>(cls + ((p.max_jobs + SEG + 15) & ~static_cast<i64>(15)));
  // two lists of (s, o) pairs for windows of which fewer than half of the positions still take part
  uint2* const list0 = reinterpret_cast<uint2*>(reinterpret_cast<unsigned char*>(G) + ((static_cast<size_t>(p.max_jobs) / SEG + 2) * MAXP * 4));
  uint2* const list1 = list0 + (p.max_jobs + 1);
  u32* const fin_start = reinterpret_cast<u32*>(p.fin_rank) + static_cast<i64>(blockIdx.x) * p.max_jobs;
  // bounds of the scratch parts, for the checked build
  const int cls_cap = static_cast<int>((p.max_jobs + SEG + 15) & ~static_cast<i64>(15));       // bytes
  const int g_cap = static_cast<int>((static_cast<size_t>(p.max_jobs) / SEG + 2) * MAXP);       // words
  const int list_cap = static_cast<int>(p.max_jobs + 1);                                        // (s, o) pairs per list
  const int z_cap = static_cast<int>(KVS_CTA_SCRATCH(p.max_jobs) / 4);                          // words of the whole block
  (void)cls_cap; (void)g_cap; (void)list_cap; (void)z_cap;
  if (!LIGHT) {
    for (int i = tid; i < RINGW; i += T) { sh.dA[i] = 0; sh.dB[i] = 0; }
  }

  for (;;) {
    __syncthreads();
    if (tid == 0) {
      sh.next_eval = static_cast<i64>(atomicAdd(p.counter, 1ull));
      sh.fallback = 0;
      sh.n_runs = 0;
    }
    __syncthreads();
    // A call with few evaluations shares each of them between `parts` CTAs: all of them form the plan (its scratch is
    // the CTA's own), each takes a share of the job results and, since the phases' rounds are disjoint, walks a range of
    // phases of about equal cost; the CTA that finishes last writes the scalars.
    constexpr bool SHARED = FAM == KVS_FUSED_SHARED || FAM == KVS_FUSED_SHARED_EST;
    const int all_parts = SHARED ? p.parts : 1;
    const int my_part = SHARED ? static_cast<int>(sh.next_eval % all_parts) : 0;
    const i64 slot_no = SHARED ? sh.next_eval / all_parts : sh.next_eval;
    if (slot_no >= (p.eval_list ? static_cast<i64>(*p.eval_count) : p.P)) break;
    const i64 e = p.eval_list ? p.eval_list[slot_no] : slot_no;
    const kvs_setting st = p.settings[e];
    const i64 lo = p.job_off[st.instance];
    const InstStats stats = p.stats[st.instance];
    const int n = stats.flags ? 0 : static_cast<int>(p.job_off[st.instance + 1] - lo);
    const i64 M = st.M;
    const i64 s_bar = st.s_bar >= 0 ? st.s_bar : stats.s_max;
    const i64 X = M - s_bar;
    const int family = FAM < 0 ? st.family : FAM;
    const bool geometric = family == KVS_GBA || family == KVS_GSA;
    const bool sim = family == KVS_SIMS;
    const bool batches = VARIANTS && geometric && st.subroutine == 1;      // simultaneous batches inside the phases
    const bool per_class = VARIANTS && geometric && st.per_class_s == 1;   // parallelism from the longest prompt of a phase
    const bool slots = sim || batches;                         // runs start together, k of them at a time
    const bool est = FAM == KVS_FUSED_SHARED_EST || (FAM == KVS_FUSED_ANY && p.key != nullptr);
    const bool keyed = !(family == KVS_GSA && !est);          // plain GSA keeps the index order
    const bool carry = geometric && (family == KVS_GSA || est);
    const bool est_class = est && family == KVS_GBA;          // classes by the clipped estimate
    const bool pow2 = geometric && st.alpha_num == 2 && st.alpha_den == 1 && st.beta0 <= 0;
    // arrays in schedule order (of the instance)
    const int32_t* const S_ord = (keyed ? p.sorted_s : p.s) + lo;
    const int32_t* const O_ord = (keyed ? p.sorted_o : p.o) + lo;
    const int32_t* const K_ord = est ? p.sorted_key + lo : O_ord;
    const int32_t* const IPERM = keyed ? p.iperm + lo : nullptr;
    const int32_t* const O_JOB = p.o + lo;
    const i64* const ARR = p.arrival ? p.arrival + lo : nullptr;
    const i64 job_out = p.out.job_out_off ? p.out.job_out_off[e] : 0;
    int32_t* const out_start = p.out.job_start ? p.out.job_start + job_out : nullptr;
    int32_t* const out_done = p.out.job_completion ? p.out.job_completion + job_out : nullptr;
    const i64 prof_base = p.ev.profile_off ? p.ev.profile_off[e] : 0;
    const i64 prof_cap = (p.ev.profile && p.ev.profile_off) ? p.ev.profile_off[e + 1] - prof_base : 0;
    int32_t* const prof = p.ev.profile ? p.ev.profile + prof_base : nullptr;
    if (geometric && (st.subroutine == 1 || st.per_class_s == 1) && (!VARIANTS || est || (p.do_profile && prof_cap > 0))) {
      // these variants on estimates, and their profiles, are the general kernel's
      if (tid == 0 && my_part == 0) p.slow_list[atomicAdd(p.slow_count, 1ull)] = e;
      continue;
    }
    const bool want32 = p.out.job_start || p.out.job_completion;
    const bool event_form = p.do_profile && !geometric && p.prefix_s != nullptr && prof_cap == 0;
    // Batching on exact keys with no profile wanted: a class is an SPS schedule in key order, its peak comes from run ends too.
    const bool class_form = p.do_profile && family == KVS_GBA && !est && prof_cap == 0;
    const bool walk = p.do_profile && !event_form && !class_form;     // rounds are walked tile by tile
    if (LIGHT && walk) {
      if (tid == 0) p.walk_list[atomicAdd(p.walk_count, 1ull)] = e;
      continue;
    }

    int status = stats.flags;
    // a block of per-job results that does not hold the instance's jobs is not written
    if (!status && (p.out.job_start || p.out.job_completion) && p.out.job_out_off[e + 1] - job_out < n) status = KVS_EVAL_CAPACITY | KVS_EVAL_BAD_INPUT;
    if (!status && (X < 1 || stats.o_max > X)) status = KVS_EVAL_INFEASIBLE;
    if (!status && geometric) {
      if (tid < 32) ladder32(sh, X, st.alpha_num, st.alpha_den, st.beta0, static_cast<u32>(s_bar), static_cast<u32>(M), batches);
      __syncthreads();
      if (sh.n_phases == 0) status = KVS_EVAL_RANGE;
    }

    FAcc acc;
    i64 base = 0;          // first round of the next phase
    i64 written_to = 0;    // profile rounds [0, written_to) have been written
    bool give_up = false;
    u32 top = 0;           // largest memory found so far, the same in every thread (evaluations that store no profile)

    int seg_lo = 0;
    while (!status && !give_up && seg_lo < n) {
      // ---- window = offline sub-instance [seg_lo, seg_hi) ----
      if (tid < 32) {
        const int end = p.window > 0 && ARR ? window_end(ARR, seg_lo, n, p.window) : n;
        if (tid == 0) sh.seg_end = end;
      }
      __syncthreads();
      const int seg_hi = sh.seg_end;
      const int nseg = seg_hi - seg_lo;
      if (p.window > 0 && ARR) base = max_i64(base, (ARR[seg_lo] / p.window + 1) * p.window);

      int L = 1;
      if (geometric) {
        L = sh.n_phases;
        for (int q = tid; q <= L; q += T) {
          int v;
          if (q == 0) v = 0;
          else if (q == L || family == KVS_GSA) v = nseg;
          else {
            const i64 t = sh.tau[q - 1];
            int a = 0, b = nseg;
            while (a < b) { const int m = (a + b) >> 1; if (K_ord[seg_lo + m] <= t) a = m + 1; else b = m; }
            v = a;
          }
          sh.ent[q] = v;
        }
      } else if (tid == 0) {
        const i64 tau = st.tau > 0 ? st.tau : static_cast<i64>(K_ord[seg_hi - 1]);   // largest key of the segment
        i64 k = st.k;
        if (k <= 0) k = sim ? M / (s_bar + tau) : (s_bar + tau <= M ? static_cast<i64>(max_parallelism32(static_cast<u32>(tau), static_cast<u32>(s_bar), static_cast<u32>(M))) : 0);
        sh.tau[0] = static_cast<u32>(tau);
        sh.k[0] = k < 1 ? 0u : static_cast<u32>(k);
        sh.ent[0] = 0; sh.ent[1] = nseg;
      }
      __syncthreads();
      if (!geometric && sh.k[0] < 1) { status = KVS_EVAL_INFEASIBLE; break; }

      // ---- plan: participants, length and first round of every phase ----
      const u32 Xc = static_cast<u32>(X);
      const int nsegs = (nseg + SEG - 1) / SEG;
      if (carry) {
        // leaving class of every position, and per segment the number of positions that leave in
        // phase q or later (row `seg` of the table, not yet summed over the segments before it).  Counted by one byte
        // compare per lane and class that occurs: with right-skewed lengths most positions of a segment share a class,
        // which makes counting by atomics a chain of conflicts.
        for (int seg = warp; seg < nsegs; seg += WARPS) {
          const int xb = seg * SEG + 8 * lane;
          const int room = nseg - xb;
          const u32 lim = room >= 8 ? 0xffu : (room > 0 ? (1u << room) - 1u : 0u);
          u32 w0 = 0, w1 = 0, c_min = 0xffu, c_max = 0u;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int x = xb + j;
            if (x < nseg) {
              u32 v = static_cast<u32>(__ldg(O_ord + seg_lo + x));
              if (est_class) { const u32 kc = min(static_cast<u32>(__ldg(K_ord + seg_lo + x)), Xc); v = max(v, kc); }
              const u32 c = static_cast<u32>(pow2 ? class_pow2(Xc, v) : class_of(sh.tau, L, v));
              if (j < 4) w0 |= c << (8 * j); else w1 |= c << (8 * (j - 4));
              c_min = min(c_min, c); c_max = max(c_max, c);
            }
          }
          if (KVS_IN(xb + 7, cls_cap, CHK_CLS)) *reinterpret_cast<uint2*>(cls + xb) = make_uint2(w0, w1);
          const int pmin = static_cast<int>(__reduce_min_sync(0xffffffffu, c_min));
          const int pmax = static_cast<int>(__reduce_max_sync(0xffffffffu, c_max));
          const u32 all = __reduce_add_sync(0xffffffffu, static_cast<u32>(__popc(lim)));
          // lane q holds the counts of classes q, q + 32, q + 64
          u32 h0 = lane <= pmin ? all : 0u, h1 = lane + 32 <= pmin ? all : 0u, h2 = lane + 64 <= pmin ? all : 0u;
          for (int q = pmin + 1; q <= pmax; ++q) {
            const u32 p4 = static_cast<u32>(q) * 0x01010101u;
            const u32 ge = (byte_mask4(w0, p4, true) | byte_mask4(w1, p4, true) << 4) & lim;
            const u32 c = __reduce_add_sync(0xffffffffu, static_cast<u32>(__popc(ge)));
            if (lane == (q & 31)) { if (q < 32) h0 = c; else if (q < 64) h1 = c; else h2 = c; }
          }
          if (KVS_IN(seg * L + L - 1, g_cap, CHK_G)) {
            if (lane < L) G[seg * L + lane] = h0;
            if (lane + 32 < L) G[seg * L + lane + 32] = h1;
            if (lane + 64 < L) G[seg * L + lane + 64] = h2;
          }
        }
        __syncthreads();
        // exclusive sums over the segments; row nsegs = totals
        const int rpw = (nsegs + WARPS - 1) / WARPS;
        const int sa = min(nsegs, warp * rpw), sb = KVS_IN(nsegs * L + L - 1, g_cap, CHK_G) ? min(nsegs, sa + rpw) : sa;
        u32 a0 = 0, a1 = 0, a2 = 0;
        for (int seg = sa; seg < sb; ++seg) {
          if (lane < L) a0 += G[seg * L + lane];
          if (lane + 32 < L) a1 += G[seg * L + lane + 32];
          if (lane + 64 < L) a2 += G[seg * L + lane + 64];
        }
        sh.cnt[warp][lane] = a0; sh.cnt[warp][lane + 32] = a1; sh.cnt[warp][lane + 64] = a2;
        __syncthreads();
        u32 r0 = 0, r1 = 0, r2 = 0;
        for (int w = 0; w < warp; ++w) { r0 += sh.cnt[w][lane]; r1 += sh.cnt[w][lane + 32]; r2 += sh.cnt[w][lane + 64]; }
        for (int seg = sa; seg < sb; ++seg) {
          if (lane < L) { const u32 t = G[seg * L + lane]; G[seg * L + lane] = r0; r0 += t; }
          if (lane + 32 < L) { const u32 t = G[seg * L + lane + 32]; G[seg * L + lane + 32] = r1; r1 += t; }
          if (lane + 64 < L) { const u32 t = G[seg * L + lane + 64]; G[seg * L + lane + 64] = r2; r2 += t; }
        }
        if (warp == WARPS - 1 && KVS_IN(nsegs * L + L - 1, g_cap, CHK_G)) {
          // positions that leave in phase q or later: all of them take part in q once they have entered
          if (lane < L) { G[nsegs * L + lane] = r0; sh.np[lane] = r0; }
          if (lane + 32 < L) { G[nsegs * L + lane + 32] = r1; sh.np[lane + 32] = r1; }
          if (lane + 64 < L) { G[nsegs * L + lane + 64] = r2; sh.np[lane + 64] = r2; }
        }
        __syncthreads();
      }
      if (per_class) {
        // longest prompt among a phase's participants: of the class itself, and under slicing of the later classes too
        for (int q = tid; q < L; q += T) sh.s_top[q] = 0;
        __syncthreads();
        for (int x = tid; x < nseg; x += T) {
          const int c = carry ? static_cast<int>(KVS_IN(x, cls_cap, CHK_CLS) ? cls[x] : 0) : class_of(sh.tau, L, static_cast<u32>(__ldg(O_ord + seg_lo + x)));
          const u32 s = static_cast<u32>(__ldg(S_ord + seg_lo + x));
          if (s > *const_cast<volatile u32*>(&sh.s_top[c])) atomicMax(&sh.s_top[c], s);
        }
        __syncthreads();
        if (tid < L) {
          u32 s = sh.s_top[tid];
          if (carry)
            for (int q = tid + 1; q < L; ++q) s = max(s, sh.s_top[q]);
          const u32 tau = sh.tau[tid];
          u32 k = 0;
          if (static_cast<i64>(s) + tau <= M) k = batches ? static_cast<u32>(M / (static_cast<i64>(s) + tau)) : max_parallelism32(tau, s, static_cast<u32>(M));
          sh.k[tid] = max(k, 1u);
          // not one of the phase's jobs fits: the general kernel reports it
          if (k < 1 && (carry ? sh.ent[tid + 1] - nseg + static_cast<int>(sh.np[tid]) : sh.ent[tid + 1] - sh.ent[tid]) > 0) sh.fallback = 1;
        }
        __syncthreads();
      }
      if (tid < L) {
        // entered by phase tid: positions below ent[tid + 1]; of those, the ones that leave in tid or later
        const u32 N = carry ? static_cast<u32>(sh.ent[tid + 1]) - static_cast<u32>(nseg) + sh.np[tid]
                            : static_cast<u32>(sh.ent[tid + 1] - sh.ent[tid]);
        sh.np[tid] = N;
        const u32 tau = sh.tau[tid], k = sh.k[tid];
        i64 len = 0;
        if (N > 0) len = (slots ? static_cast<i64>(ceil_div_u(N, k) - 1) * tau : static_cast<i64>(static_cast<u64>(N - 1) * tau / k)) + tau;
        sh.plen[tid] = len;
        sh.kinv[tid] = k >= 2 ? ~0ull / k + 1ull : 0ull;
        // memory is kept modulo 2^32: the general kernel reports evaluations whose bound reaches that
        if (p.do_profile && N > 0 && min_i64(N, static_cast<i64>(k) + 1) * (static_cast<i64>(stats.s_max) + tau) >= (static_cast<i64>(1) << 32))
          sh.fallback = 1;
      }
      __syncthreads();
      if (tid == 0) {
        i64 b = base, runs = sh.n_runs;
        u64 tp = 0;
        for (int q = 0; q < L; ++q) {
          sh.taupre[q] = tp;
          tp += sh.tau[q];
          sh.pbase[q] = static_cast<u32>(b);
          b += sh.plen[q];
          runs += sh.np[q];
          if (b >= TIME_LIMIT) { sh.fallback = 1; break; }
        }
        sh.taupre[L] = tp;
        sh.base_next = b;
        sh.n_runs = runs;
      }
      __syncthreads();
      if (sh.fallback) { give_up = true; break; }

      // A window of few of the jobs goes as a whole to the CTA whose part of the positions it lies in; a larger one is shared.
      int parts = all_parts, part = my_part;
      if (SHARED && all_parts > 1 && 2 * static_cast<i64>(nseg) * all_parts <= n) {
        if ((seg_lo + nseg / 2) * static_cast<i64>(all_parts) / n != my_part) {
          base = written_to = sh.base_next;
          seg_lo = seg_hi;
          continue;
        }
        parts = 1;
        part = 0;
      }

      // ---- per-job results ----
      if (!carry) {
        // exactly one run per job; the rank is the position inside the class.  Four jobs per thread
        // and step, loads first, so that enough memory requests are in flight.
        const u32 tau0 = sh.tau[0];
        constexpr int JU = 4;
        for (int j0 = seg_lo + tid + part * (JU * T); j0 < seg_hi; j0 += JU * T * parts) {
          u32 oj_[JU];
          int pos_[JU];
#pragma unroll
          for (int u = 0; u < JU; ++u) {
            const int j = j0 + u * T;
            oj_[u] = 0; pos_[u] = 0;
            if (j < seg_hi) {
              oj_[u] = static_cast<u32>(__ldg(O_JOB + j));
              pos_[u] = IPERM ? __ldg(IPERM + j) : j;
            }
          }
#pragma unroll
          for (int u = 0; u < JU; ++u) {
            const int j = j0 + u * T;
            if (j >= seg_hi) break;
            const u32 oj = oj_[u];
            int ph = 0;
            bool fin = true;
            if (geometric) ph = pow2 ? class_pow2(Xc, oj) : class_of(sh.tau, L, oj);
            else fin = oj <= tau0;
            const u32 rank = static_cast<u32>(pos_[u] - seg_lo - sh.ent[ph]);
            const u32 tau = sh.tau[ph], k = sh.k[ph];
            const u32 stt = sh.pbase[ph] + (slots ? (rank / k) * tau : slot_mul(rank, tau, k, sh.kinv[ph]));
            const u32 d = fin ? oj : tau;
            acc.steps += d;
            acc.hmax = max(acc.hmax, stt + d);
            int32_t start = -1, done = -1;
            if (fin) {
              start = static_cast<int32_t>(stt);
              done = static_cast<int32_t>(stt + oj);
              acc.flow += static_cast<u64>(static_cast<i64>(done) - (ARR ? __ldg(ARR + j) : 0));
            } else {
              ++acc.unfinished;
            }
            if (!KVS_IN(j, n, CHK_JOB_OUT)) continue;
            if (out_start) __stcs(&out_start[j], start);
            if (out_done) __stcs(&out_done[j], done);
          }
        }
      } else {
        // The rank of a job in the phase that completes it = positions before it that leave in that
        // phase or later: the table gives the count before the segment; inside the segment a lane
        // holds the classes of eight consecutive positions, and for every class q present one byte
        // compare per lane and one warp scan count the positions with class >= q before each lane.
        const bool vec_o = (reinterpret_cast<uintptr_t>(O_ord + seg_lo) & 15u) == 0;
        // (keyed: the start rounds pass through the CTA's own scratch, so a shared evaluation forms them all in every CTA)
        for (int seg = keyed ? warp : warp + WARPS * part; seg < nsegs; seg += keyed ? WARPS : WARPS * parts) {
          const int xb = seg * SEG + 8 * lane;
          const int room = nseg - xb;
          const u32 lim = room >= 8 ? 0xffu : (room > 0 ? (1u << room) - 1u : 0u);
          u32 ov_[8];
          if (vec_o && room >= 8) {
            const uint4 b0 = __ldg(reinterpret_cast<const uint4*>(O_ord + seg_lo + xb));
            const uint4 b1 = __ldg(reinterpret_cast<const uint4*>(O_ord + seg_lo + xb) + 1);
            ov_[0] = b0.x; ov_[1] = b0.y; ov_[2] = b0.z; ov_[3] = b0.w; ov_[4] = b1.x; ov_[5] = b1.y; ov_[6] = b1.z; ov_[7] = b1.w;
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) ov_[j] = (lim >> j & 1u) ? static_cast<u32>(__ldg(O_ord + seg_lo + xb + j)) : 0u;
          }
          const uint2 cw = KVS_IN(xb + 7, cls_cap, CHK_CLS) ? *reinterpret_cast<const uint2*>(cls + xb) : make_uint2(0, 0);
          // smallest and largest class among the warp's valid positions
          u32 lo4 = 0xffu, hi4 = 0u;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const u32 c = ((j < 4 ? cw.x : cw.y) >> (8 * (j & 3))) & 0xffu;
            if (lim >> j & 1u) { lo4 = min(lo4, c); hi4 = max(hi4, c); }
          }
          const int pmin = static_cast<int>(__reduce_min_sync(0xffffffffu, lo4));
          const int pmax = static_cast<int>(__reduce_max_sync(0xffffffffu, hi4));
          u32 rk_[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) rk_[j] = 0;
          for (int q = pmin; q <= pmax; ++q) {
            const u32 p4 = static_cast<u32>(q) * 0x01010101u;
            const u32 ge = (byte_mask4(cw.x, p4, true) | byte_mask4(cw.y, p4, true) << 4) & lim;
            const u32 eq = (byte_mask4(cw.x, p4, false) | byte_mask4(cw.y, p4, false) << 4) & lim;
            const u32 cnt = static_cast<u32>(__popc(ge));
            u32 incl = cnt;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
              const u32 y = __shfl_up_sync(0xffffffffu, incl, d);
              if (lane >= d) incl += y;
            }
            if (eq) {
              const u32 before = (KVS_IN(seg * L + q, g_cap, CHK_G) ? G[seg * L + q] : 0u) + incl - cnt;
#pragma unroll
              for (int j = 0; j < 8; ++j)
                if (eq >> j & 1u) rk_[j] = before + static_cast<u32>(__popc(ge & ((1u << j) - 1u)));
            }
          }
          u32 st_[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            st_[j] = 0;
            if (lim >> j & 1u) {
              const int l = static_cast<int>(((j < 4 ? cw.x : cw.y) >> (8 * (j & 3))) & 0xffu);
              int f = 0;
              if (est_class) {
                const u32 kc = min(static_cast<u32>(__ldg(K_ord + seg_lo + xb + j)), Xc);
                f = pow2 ? class_pow2(Xc, kc) : class_of(sh.tau, L, kc);
              }
              const u32 tau = sh.tau[l], k = sh.k[l];
              st_[j] = sh.pbase[l] + (batches ? (rk_[j] / k) * tau : slot_mul(rk_[j], tau, k, sh.kinv[l]));
              if (!SHARED || !keyed || (seg / WARPS) % parts == part) acc.steps += ov_[j] + (sh.taupre[l] - sh.taupre[f]);
            }
          }
          if (keyed) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if ((lim >> j & 1u) && KVS_IN(seg_lo + xb + j, p.max_jobs, CHK_FIN)) fin_start[seg_lo + xb + j] = st_[j];
          } else {
            if (room > 0 && !KVS_IN(seg_lo + xb + min(room, 8) - 1, n, CHK_JOB_OUT)) continue;
            const bool vec_out = room >= 8 && ((seg_lo + xb) & 3) == 0 &&
                                 ((reinterpret_cast<uintptr_t>(out_start) | reinterpret_cast<uintptr_t>(out_done)) & 15u) == 0;
            u32 dn_[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              dn_[j] = st_[j] + ov_[j];
              if (lim >> j & 1u) {
                acc.hmax = max(acc.hmax, dn_[j]);
                acc.flow += static_cast<u64>(static_cast<i64>(dn_[j]) - (ARR ? __ldg(ARR + seg_lo + xb + j) : 0));
              }
            }
            if (vec_out) {
              if (out_start) {
                int4* const d = reinterpret_cast<int4*>(out_start + seg_lo + xb);
                __stcs(d, make_int4(static_cast<int>(st_[0]), static_cast<int>(st_[1]), static_cast<int>(st_[2]), static_cast<int>(st_[3])));
                __stcs(d + 1, make_int4(static_cast<int>(st_[4]), static_cast<int>(st_[5]), static_cast<int>(st_[6]), static_cast<int>(st_[7])));
              }
              if (out_done) {
                int4* const d = reinterpret_cast<int4*>(out_done + seg_lo + xb);
                __stcs(d, make_int4(static_cast<int>(dn_[0]), static_cast<int>(dn_[1]), static_cast<int>(dn_[2]), static_cast<int>(dn_[3])));
                __stcs(d + 1, make_int4(static_cast<int>(dn_[4]), static_cast<int>(dn_[5]), static_cast<int>(dn_[6]), static_cast<int>(dn_[7])));
              }
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                if (lim >> j & 1u) {
                  if (out_start) __stcs(&out_start[seg_lo + xb + j], static_cast<int32_t>(st_[j]));
                  if (out_done) __stcs(&out_done[seg_lo + xb + j], static_cast<int32_t>(dn_[j]));
                }
              }
            }
          }
        }
        if (keyed) {
          __syncthreads();
          for (int j = seg_lo + tid + part * T; j < seg_hi; j += T * parts) {
            const u32 oj = static_cast<u32>(__ldg(O_JOB + j));
            const int ip = __ldg(IPERM + j);
            if (!KVS_IN(ip, p.max_jobs, CHK_FIN) || !KVS_IN(j, n, CHK_JOB_OUT)) continue;
            const u32 stt = fin_start[ip];
            const u32 done = stt + oj;
            acc.hmax = max(acc.hmax, done);
            acc.flow += static_cast<u64>(static_cast<i64>(done) - (ARR ? __ldg(ARR + j) : 0));
            if (out_start) __stcs(&out_start[j], static_cast<int32_t>(stt));
            if (out_done) __stcs(&out_done[j], static_cast<int32_t>(done));
          }
        }
      }

      // ---- memory profile ----
      if (event_form && part == 0) {
        // SPS / SimS in exact key order with no profile wanted: the peak comes from the run ends
        // (see kvs_events.cuh for why the last round of every run is enough), here in 32-bit
        // arithmetic, which the bound checked by the plan makes exact.
        const u32* const ps32 = reinterpret_cast<const u32*>(p.prefix_s + lo + st.instance + seg_lo);   // low words
        const u32 tau = sh.tau[0], k = sh.k[0];
        const u32 N = static_cast<u32>(nseg);
        const int32_t* const Ow = O_ord + seg_lo;
        if (sim) {
          // a batch is alone in its slot: in the last round of run i the jobs i .. end of the batch
          // are active with progress d_i - 1
          for (u32 i0 = tid; i0 < N; i0 += 4 * T) {
            u32 o_[4], p_[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const u32 i = i0 + u * T;
              o_[u] = i < N ? static_cast<u32>(__ldg(Ow + i)) : 0u;
              p_[u] = i < N ? ps32[2 * static_cast<size_t>(i)] : 0u;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const u32 i = i0 + u * T;
              if (i < N) {
                const u32 bend = min(N, (i / k + 1u) * k);
                const u32 d = min(o_[u], tau);
                acc.peak = max(acc.peak, ps32[2 * static_cast<size_t>(bend)] - p_[u] + (bend - i) * d);
              }
            }
          }
        } else {
          // Z[m] = sum over ranks j < m of (s_j - start_j): the jobs [i, b) active in round t hold
          // Z[b] - Z[i] + (b - i)(t + 1) tokens.  First Z for every rank, then one candidate per run.
          // four ranks per thread and step: shorter dependent chains than the ring's rounds per thread
          constexpr int EVI = 4;
          u32* const Z = reinterpret_cast<u32*>(cls);      // N + 1 words of this CTA's scratch
          const u32 qt = tau / k, rt = tau - qt * k;
          u32 F_run = 0;
          for (u32 c0 = 0; c0 <= N; c0 += (T * EVI)) {
            const u32 r = c0 + EVI * tid;
            u32 q = 0, rem = 0;
            if (r <= N) { u64 dq_, dr_; divmod_u(static_cast<u64>(r) * tau, k, &dq_, &dr_); q = static_cast<u32>(dq_); rem = static_cast<u32>(dr_); }
            u32 f[EVI], tot = 0;
#pragma unroll
            for (int j = 0; j < EVI; ++j) {
              f[j] = tot;
              if (r + j < N) tot += q;
              rem += rt; q += qt;
              if (rem >= k) { rem -= k; ++q; }
            }
            u32 incl = tot;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
              const u32 y = __shfl_up_sync(0xffffffffu, incl, d);
              if (lane >= d) incl += y;
            }
            __syncthreads();
            if (lane == 31) sh.redA[warp] = incl;
            __syncthreads();
            const u32 w = lane < WARPS ? sh.redA[lane] : 0u;
            u32 wi = w;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
              const u32 y = __shfl_up_sync(0xffffffffu, wi, d);
              if (lane >= d) wi += y;
            }
            const u32 off = F_run + __shfl_sync(0xffffffffu, wi - w, warp) + (incl - tot);
            F_run += __shfl_sync(0xffffffffu, wi, 31);
#pragma unroll
            for (int j = 0; j < EVI; ++j)
              if (r + j <= N && KVS_IN(r + j, z_cap, CHK_Z)) Z[r + j] = ps32[2 * static_cast<size_t>(r + j)] - (off + f[j]);
          }
          __syncthreads();
          for (u32 c0 = 0; c0 < N; c0 += (T * EVI)) {
            const u32 r = c0 + EVI * tid;
            if (r >= N) continue;
            u64 dq_, dr_;
            divmod_u(static_cast<u64>(r) * tau, k, &dq_, &dr_);
            u32 q = static_cast<u32>(dq_), rem = static_cast<u32>(dr_);
            u32 o_[EVI], z_[EVI];
#pragma unroll
            for (int j = 0; j < EVI; ++j) {
              o_[j] = r + j < N ? static_cast<u32>(__ldg(Ow + r + j)) : 0u;
              z_[j] = (r + j < N && KVS_IN(r + j, z_cap, CHK_Z)) ? Z[r + j] : 0u;
            }
#pragma unroll
            for (int j = 0; j < EVI; ++j) {
              if (r + j < N) {
                const u32 t1 = q + min(o_[j], tau);                       // last round of the run, plus one
                const u64 x = static_cast<u64>(t1) * k + (tau - 1u);      // b = ranks that start before t1
                const u32 b = (x >> 32) ? static_cast<u32>(min(static_cast<u64>(N), x / tau)) : min(N, static_cast<u32>(x) / tau);
                if (KVS_IN(b, z_cap, CHK_Z)) acc.peak = max(acc.peak, Z[b] - z_[j] + (b - (r + j)) * t1);
              }
              rem += rt; q += qt;
              if (rem >= k) { rem -= k; ++q; }
            }
          }
          __syncthreads();     // Z is scratch of the next window too
        }
      } else if (class_form) {
        // Per class, Z[m] = sum over its ranks j < m of (s_j - start_j); in the last round of run i, whose end no later run's
        // precedes, the ranks [i, b) that have started hold Z[b] - Z[i] + (b - i)(t + 1) tokens (kvs_events.cuh).
        u32* const Z = reinterpret_cast<u32*>(cls);
        for (int ph = 0; ph < L; ++ph) {
          const int N = static_cast<int>(sh.np[ph]);
          if (N == 0 || (parts > 1 && ph % parts != part)) continue;
          const int32_t* const Sc = S_ord + seg_lo + sh.ent[ph];
          const int32_t* const Oc = O_ord + seg_lo + sh.ent[ph];
          const u32 tau = sh.tau[ph], k = sh.k[ph];
          const u64 kinv = sh.kinv[ph];
          if (batches) {
            // a batch is alone in its slot: in the last round of run i the jobs i .. end of the batch are active
            block_prefix(sh, Z, z_cap, N, [&](int r) { return static_cast<u32>(__ldg(Sc + r)); });
            for (u32 r = tid; r < static_cast<u32>(N); r += T) {
              const u32 bend = batch_end(r, k, N);
              if (KVS_IN(bend, z_cap, CHK_Z)) acc.peak = max(acc.peak, Z[bend] - Z[r] + (bend - r) * static_cast<u32>(__ldg(Oc + r)));
            }
            __syncthreads();
            continue;
          }
          block_prefix(sh, Z, z_cap, N, [&](int r) { return static_cast<u32>(__ldg(Sc + r)) - slot_mul(static_cast<u32>(r), tau, k, kinv); });
          for (int r = tid; r < N; r += T) {
            const u32 t1 = slot_mul(static_cast<u32>(r), tau, k, kinv) + static_cast<u32>(__ldg(Oc + r));
            const u64 x = static_cast<u64>(t1) * k + (tau - 1u);
            const u32 b = (x >> 32) ? static_cast<u32>(min(static_cast<u64>(N), x / tau)) : min(static_cast<u32>(N), static_cast<u32>(x) / tau);
            if (KVS_IN(b, z_cap, CHK_Z)) acc.peak = max(acc.peak, Z[b] - Z[r] + (b - static_cast<u32>(r)) * t1);
          }
          __syncthreads();
        }
      } else if (!LIGHT && walk) {
        bool list_mode = false;
        uint2* cur = list0;
        uint2* nxt = list1;
        int C = 0;
        // index order without estimates: the phases before the first class that holds a job are
        // walked from prefix sums of s + 1 over the positions (see pure_phase_events)
        int n_pure = 0;
        u32* const PS = reinterpret_cast<u32*>(list1);
        if (carry && !est) {
          while (n_pure + 1 < L && static_cast<int>(sh.np[n_pure + 1]) == nseg) ++n_pure;
        }
        bool any_pure = n_pure > 0;
        // No profile stored: only the peak is wanted.  The phases are then taken from the last one back - slices grow along
        // the ladder and with them the memory held - and a phase whose upper bound does not exceed the largest memory
        // found so far is not looked at.
        // (Calls with estimates have many windows of few jobs: forming the bounds costs what the rounds do, 1,380 against 1,110 us
        // for 64 instances of 50,000 jobs.)
        const bool peak_only = prof_cap == 0 && !est;
        if (SHARED && parts > 1 && !peak_only) {
          // This CTA's share: the tiles whose middle falls into its part of the evaluation's cost; a phase of a few tiles goes
          // as a whole.  A tile costs about as much as visiting 2,048 runs, whatever starts in it; the phases walked from
          // prefix sums visit none.
          if (warp == 0) {
            i64 cost[MAXP / 32], incl[MAXP / 32], total = 0;
#pragma unroll
            for (int u = 0; u < MAXP / 32; ++u) {
              const int q = 32 * u + lane;
              cost[u] = q < L ? ((sh.plen[q] + TILE - 1) / TILE) * 2048 + (q < n_pure ? 0 : static_cast<i64>(sh.np[q])) : 0;
              const i64 v = warp_incl(cost[u]);
              incl[u] = total + v;
              total += __shfl_sync(0xffffffffu, v, 31);
            }
            const i64 lo_cost = total * part / parts, hi_cost = total * (part + 1) / parts;
#pragma unroll
            for (int u = 0; u < MAXP / 32; ++u) {
              const int q = 32 * u + lane;
              if (q >= L) continue;
              const i64 before = incl[u] - cost[u];
              const int n_tiles = static_cast<int>((sh.plen[q] + ((prof_base + sh.pbase[q]) & 3) + TILE - 1) / TILE);
              const int grain = n_tiles < 6 ? 1 : n_tiles;
              auto first_at = [&](i64 x) {         // first of `grain` pieces whose middle is at or after x
                if (x <= before || cost[u] == 0) return 0;
                if (x >= incl[u]) return grain;
                // middle of piece i: (2 i + 1) / (2 grain) of the cost
                return static_cast<int>(min_i64(grain, ceil_div_u(static_cast<u64>(2 * (x - before)) * grain, static_cast<u64>(cost[u])) / 2));
              };
              sh.tile_lo[q] = grain == 1 ? first_at(lo_cost) * n_tiles : first_at(lo_cost);
              sh.tile_hi[q] = part == parts - 1 ? n_tiles : (grain == 1 ? first_at(hi_cost) * n_tiles : first_at(hi_cost));
            }
          }
          __syncthreads();
          bool mine = false;
          for (int q = tid; q < n_pure; q += T) mine |= sh.tile_lo[q] < sh.tile_hi[q];
          any_pure = __syncthreads_or(mine) != 0;
        }
        bool begun = false;
        int turn = 0;
        auto s_plus_1 = [&](int x) { return static_cast<u32>(__ldg(S_ord + seg_lo + x)) + 1u; };
        if (carry && !est) {
          if (any_pure && !peak_only) block_prefix(sh, PS, 2 * list_cap, nseg, s_plus_1);
        }
        bool have_ps = !peak_only;               // prefix sums over positions; a peak-only evaluation forms them when it needs them
        u32 pure_widest = 0;
        for (int it = 0; it < L; ++it) {
          const int ph = peak_only ? L - 1 - it : it;
          const int N = static_cast<int>(sh.np[ph]);
          if (N == 0) continue;
          int part_of = 0, parts_of = 1;           // share of a phase that all CTAs of the evaluation look at
          // tile origins keep the profile stores 16-byte aligned
          const int a0 = -static_cast<int>((prof_base + sh.pbase[ph]) & 3);
          const int n_tiles = static_cast<int>((sh.plen[ph] - a0 + TILE - 1) / TILE);
          int tile_lo = 0, tile_hi = n_tiles;
          if (SHARED && parts > 1 && peak_only) {
            // The phases are taken in turn, but one of many pairs of run ends and runs is looked at by all CTAs, each of which takes a
            // share of its run ends: 64 initial slices on 20,000 jobs, whose longest evaluations have few phases, 331 -> 237 us.
            const u64 pairs = static_cast<u64>(N) * min(static_cast<u32>(N), sh.k[ph]), rounds = static_cast<u64>(n_tiles) * 6000;
            if (!batches && !sim && ph >= n_pure && pairs > SHARED_PAIRS && rounds >= static_cast<u64>(N) && pairs / T * PAIR_CYCLES / parts < rounds) { part_of = part; parts_of = parts; }
            else if (turn++ % parts != part) continue;
            // what the other CTAs of this evaluation have found
            __syncthreads();
            if (tid == 0) sh.redA[0] = atomicMax(&p.shares[slot_no].peak, top);
            __syncthreads();
            top = max(top, sh.redA[0]);
            __syncthreads();
          } else if (SHARED && parts > 1) {
            tile_lo = sh.tile_lo[ph];
            tile_hi = sh.tile_hi[ph];
            // idle rounds before the window's first phase are the first share's; later phases follow one another
            if (!begun && part == 0 && prof_cap > 0)
              for (i64 t = written_to + tid; t < sh.pbase[ph] && t < prof_cap; t += T) prof[t] = 0;
            begun = true;
            written_to = sh.pbase[ph];
            if (tile_lo >= tile_hi) continue;
          }
          PhaseView P;
          P.S = S_ord + seg_lo; P.O = O_ord + seg_lo;
          P.cls = cls; P.G = G; P.L = L; P.ph = ph; P.nsegs = nsegs;
          P.cls_cap = cls_cap; P.g_cap = g_cap;
          P.gcol = nullptr;
          P.n_src = nseg;
          P.x_lo = carry ? 0 : sh.ent[ph];
          P.x_hi = sh.ent[ph + 1];
          P.tau = sh.tau[ph]; P.k = sh.k[ph];
          P.qt = P.tau / P.k; P.rt = P.tau - P.qt * P.k;
          P.len = static_cast<u32>(sh.plen[ph]);
          P.base = sh.pbase[ph];
          const bool thin = static_cast<u64>(TILE) * P.k < 2ull * T * P.tau;     // fewer than two runs per thread and tile
          const bool dense = !sim && P.tau < TILE && P.k >= 4 * P.tau;
          ListView V;
          V.cur = cur; V.C = C; V.src = sh.ent[ph]; V.cap = list_cap;
          if (peak_only && !sim) {
            const bool pure = ph < n_pure, listed = carry && !pure;
            const bool few = 2 * N <= nseg || thin;
            // Phases of short slices in which most jobs take part, eight or more of whose runs start per round: visiting them takes
            // about a cycle per run, little more than forming the bound, and needs no list (1,024 instances of 20,000 jobs from host memory 3,702 -> 3,374 us).
            const bool sliced = listed && !few && !batches && P.tau < static_cast<u32>(TILE) && P.k >= 8u * P.tau;
            const bool straight = sliced && static_cast<u64>(n_tiles) * 6000 < static_cast<u64>(N);
            if (listed && !straight) { list_participants(P, cur, list_cap); V.C = N; }
            const u32 kk = min(static_cast<u32>(N), P.k);
            if (batches) {
              if (pure) {
                // nobody leaves: a batch holds the most in the last round of its slot (these phases come last: one prefix sum)
                if (!have_ps) block_prefix(sh, PS, 2 * list_cap, nseg, s_plus_1);
                have_ps = true;
                acc.peak = max(acc.peak, widest_batch(PS, 2 * list_cap, N, kk, P.tau - 1u));
                continue;
              }
              block_prefix(sh, PS, 2 * list_cap, N, [&](int r) { return cur[r].x; });
              // every participant runs for more than the slice before
              const u32 low = ph > 0 ? min(sh.tau[ph - 1], P.tau - 1u) : 0u;
              if (block_max(widest_batch(PS, 2 * list_cap, N, kk, P.tau), sh.redA, 0u) <= top) continue;
              acc.peak = max(acc.peak, batches_peak(sh, cur, PS, list_cap, N, kk, P.tau, low));
              top = max(top, block_max(acc.peak, sh.redA, 0u));
              continue;
            }
            // Upper bound: the largest sum of s over a window of kk ranks, as if no run in it had ended, and
            // sum_{x < kk} (tau - floor(x tau / k)) for the rounds they have run.
            const u64 ran = static_cast<u64>(kk) * (P.tau + 1ull) - static_cast<u64>(P.tau) * kk * (kk - 1ull) / (2ull * P.k);
            auto widest = [&](u32 w) {          // largest difference of the prefix sums over w ranks
              u32 W = 0;
              const u32 last = static_cast<u32>(N) - w;       // start of the last window
              for (u32 r0 = tid; r0 <= last; r0 += 4 * T) {
                u32 a[4], b[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  const u32 r = min(r0 + u * T, last);
                  a[u] = PS[r];
                  b[u] = KVS_IN(r + w, 2 * list_cap, CHK_PS) ? PS[r + w] : a[u];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) W = max(W, b[u] - a[u]);
              }
              return block_max(W, sh.redA, 0u);
            };
            // Cycles of a CTA, roughly: PAIR_CYCLES per step of a thread over the pairs of a run end and a run that may be active
            // then, against 6,000 per tile and 8 per run; the bound takes the prefix sums over the ranks.
            const u64 pairs = static_cast<u64>(N) * kk, by_ends = pairs / T * PAIR_CYCLES / parts_of + 1500, by_rounds = static_cast<u64>(n_tiles) * 6000 + static_cast<u64>(N) * (sliced ? 1 : 8);
            if (pure) {
              // the window of all these phases at their largest parallelism bounds each of them
              if (!have_ps) {
                block_prefix(sh, PS, 2 * list_cap, nseg, s_plus_1);
                have_ps = true;
                u32 w = 1;
                for (int q = 0; q < n_pure; ++q) w = max(w, sh.k[q]);
                pure_widest = widest(min(w, static_cast<u32>(N)));
              }
              if (static_cast<u64>(pure_widest) + ran <= top) continue;
            } else if (!straight && min(by_ends, by_rounds) > 2500ull + static_cast<u64>(N)) {
              block_prefix(sh, PS, 2 * list_cap, N, [&](int r) { return listed ? cur[r].x : static_cast<u32>(__ldg(P.S + P.x_lo + r)); });
              if (static_cast<u64>(widest(kk)) + ran <= top) continue;
            }
            if (!straight && by_ends < by_rounds) {
              u32 pk;
              if (listed) pk = ends_peak(cur, list_cap, N, P.tau, P.k, sh.kinv[ph], part_of, parts_of, [&](int r) { return KVS_IN(r, list_cap, CHK_LIST) ? cur[r] : make_uint2(0, 1); });
              else pk = ends_peak(cur, list_cap, N, P.tau, P.k, sh.kinv[ph], part_of, parts_of, [&](int r) { return make_uint2(static_cast<u32>(__ldg(P.S + P.x_lo + r)), static_cast<u32>(__ldg(P.O + P.x_lo + r))); });
              acc.peak = max(acc.peak, pk);
              top = max(top, block_max(pk, sh.redA, 0u));
              continue;
            }
            list_mode = listed && few;
          } else if (carry && !list_mode && ph >= n_pure && (2 * N <= nseg || thin)) {
            // from here on the participants are kept as a list in rank order: first this phase's
            list_participants(P, cur, list_cap);
            list_mode = true;
            V.C = N;
          }
          if (carry && !list_mode && ph >= n_pure && nsegs < GCOL) {
            // the visits of a filtered phase look its column of the rank table up again and again
            for (int seg = tid; seg <= nsegs; seg += T)
              if (KVS_IN(seg * L + ph, g_cap, CHK_G)) sh.gcol[seg] = G[seg * L + ph];
            P.gcol = sh.gcol;
            __syncthreads();
          }
          int C_next = 0;
          // idle rounds before this phase (window release) hold nothing
          if (prof_cap > 0)
            for (i64 t = written_to + tid; t < P.base && t < prof_cap; t += T) prof[t] = 0;
          u32 A_run = 0, B_run = 0;
          int r_next = 0, buf = 0;
          const int u_first = a0 + tile_lo * TILE;
          if (SHARED && tile_lo > 0) {
            // ranks that start before u_first, and those of them that may still hold memory there
            auto before = [&](i64 u) -> int {
              if (u <= 0) return 0;
              const i64 r = sim ? ceil_div_u(static_cast<u64>(u), P.tau) * P.k : ceil_div_u(static_cast<u64>(u) * P.k, P.tau);
              return static_cast<int>(min_i64(r, N));
            };
            r_next = before(u_first);
            const int ra = before(static_cast<i64>(u_first) - P.tau);
            CarryIn c;
            if (ph < n_pure) {
              c = carry_in_pure(P, PS, N, u_first);
            } else {
              if (list_mode) c = carry_in_list(sh, P, V, ra, r_next, u_first, buf);
              else if (carry) c = carry_in<true>(sh, P, sim, ra, r_next, u_first, buf);
              else c = carry_in<false>(sh, P, sim, ra, r_next, u_first, buf);
              c.A = block_sum(c.A, sh.redA);
              c.B = block_sum(c.B, sh.redB);
              __syncthreads();                     // the scan of the first tile uses the same words
            }
            A_run = c.A; B_run = c.B;
          }
          // ranks that start before offset u: ceil(u*k/tau) (SPS) or ceil(u/tau)*k (SimS); the tile
          // ends advance by TILE, so quotient and remainder are stepped
          const u64 mult = sim ? 1 : static_cast<u64>(P.k);
          const u64 utau = P.tau;
          u64 cq, cr, dq, dr;
          divmod_u(static_cast<u64>(u_first + TILE) * mult, utau, &cq, &cr);
          divmod_u(static_cast<u64>(TILE) * mult, utau, &dq, &dr);
          const int u_end = SHARED && tile_hi < n_tiles ? a0 + tile_hi * TILE : static_cast<int>(P.len);
          for (int u0 = u_first; u0 < u_end; u0 += TILE) {
            const int wlen = min(TILE, static_cast<int>(P.len) - u0);
            int r_b = N;                          // the last tile takes every remaining rank
            if (u0 + TILE < static_cast<int>(P.len)) {
              const u64 rb64 = (cq + (cr > 0)) * (sim ? static_cast<u64>(P.k) : 1ull);
              if (rb64 < static_cast<u64>(N)) r_b = static_cast<int>(rb64);
            }
            cq += dq; cr += dr;
            if (cr >= utau) { cr -= utau; ++cq; }
            if (ph < n_pure) pure_phase_events(sh, P, PS, 2 * list_cap, N, u0, buf);
            else if (sim) visit_thin<true>(sh, P, r_next, r_b, u0, buf, 0);
            else if (list_mode) C_next = visit_list(sh, P, V, nxt, C_next, r_next, r_b, u0, buf, dense);
            else if (carry && P.tau < static_cast<u32>(TILE) && P.k >= 8u * P.tau) visit_runs_sliced(sh, P, r_next, r_b, u0, buf, sh.kinv[ph]);
            else if (carry) visit_runs<true>(sh, P, r_next, r_b, u0, buf, dense);
            else if (thin) visit_thin<false>(sh, P, r_next, r_b, u0, buf, sh.kinv[ph]);
            else visit_runs<false>(sh, P, r_next, r_b, u0, buf, dense);
            r_next = r_b;
            if (P.tau > TILE && ph >= n_pure) {
              if (list_mode) insert_far_ends_list(sh, P, V, N, a0, u0, wlen, buf);
              else if (carry) insert_far_ends<true>(sh, P, sim, N, a0, u0, wlen, buf);
              else insert_far_ends<false>(sh, P, sim, N, a0, u0, wlen, buf);
            }
            __syncthreads();
            scan_tile(sh, buf, static_cast<i64>(P.base) + u0, wlen, P.base, A_run, B_run, acc.peak, prof, prof_cap);
            buf ^= 1;
          }
          written_to = static_cast<i64>(P.base) + P.len;
          if (peak_only) {
            list_mode = false;
            top = max(top, block_max(acc.peak, sh.redA, 0u));
            continue;
          }
          if (list_mode) {
            __syncthreads();               // the list of killed jobs is complete before it is read
            uint2* const tmp = cur; cur = nxt; nxt = tmp;
            C = C_next;
          }
          if (SHARED && (tile_lo > 0 || tile_hi < n_tiles)) {
            // only part of the runs were visited: the next phase's participants are listed anew, and the ends that
            // lie beyond the last tile leave the ring
            list_mode = false;
            __syncthreads();
            for (int i = tid; i < RINGW; i += T) { sh.dA[i] = 0; sh.dB[i] = 0; }
            __syncthreads();
          }
        }
        if (SHARED && parts > 1) written_to = sh.base_next;
      }
      base = sh.base_next;
      seg_lo = seg_hi;
    }

    if (give_up) {
      // left to the general kernel, which writes every output of this evaluation
      if (tid == 0 && my_part == 0) p.slow_list[atomicAdd(p.slow_count, 1ull)] = e;
      continue;
    }

    if (p.fill) {
      // what this evaluation did not write: the jobs of an evaluation (or of the windows after the one) that was not
      // scheduled, and the rounds behind the last slot end
      const i64 jobs = p.out.job_out_off ? p.out.job_out_off[e + 1] - job_out : 0;
      if (out_start && my_part == 0) block_fill(out_start, static_cast<i64>(seg_lo), jobs, p.fill_job);
      if (out_done && my_part == 0) block_fill(out_done, static_cast<i64>(seg_lo), jobs, p.fill_job);
      if (prof_cap > 0 && my_part == all_parts - 1) block_fill(prof, written_to, prof_cap, p.fill_prof);
    }

    // ---- scalars ----
    i64 flow = static_cast<i64>(block_sum(acc.flow, reinterpret_cast<u64*>(sh.red64)));
    i64 steps = static_cast<i64>(block_sum(acc.steps, reinterpret_cast<u64*>(sh.red64)));
    i64 hmax = block_max(acc.hmax, sh.redA, 0u);
    int unfinished = block_sum(acc.unfinished, sh.red32);
    u32 peak32 = block_max(acc.peak, sh.redA, 0u);
    if (tid == 0) {
      if (SHARED && all_parts > 1) {
        FusedShare& s = p.shares[slot_no];
        atomicAdd(&s.flow, static_cast<ull>(flow));
        atomicAdd(&s.steps, static_cast<ull>(steps));
        atomicMax(&s.hmax, static_cast<u32>(hmax));
        atomicMax(&s.peak, peak32);
        atomicAdd(&s.unfinished, unfinished);
        __threadfence();
        if (atomicAdd(&s.done, 1u) + 1u != static_cast<u32>(all_parts)) continue;
        __threadfence();
        flow = static_cast<i64>(atomicAdd(&s.flow, 0ull));
        steps = static_cast<i64>(atomicAdd(&s.steps, 0ull));
        hmax = atomicMax(&s.hmax, 0u);
        peak32 = atomicMax(&s.peak, 0u);
        unfinished = atomicAdd(&s.unfinished, 0);
      }
      const i64 peak = static_cast<i64>(peak32);
      const bool skipped = (status & (KVS_EVAL_INFEASIBLE | KVS_EVAL_BAD_INPUT)) != 0;
      if (!skipped && prof_cap > 0 && hmax > prof_cap) status |= KVS_EVAL_CAPACITY;   // capacity 0 = profile not wanted
      const bool have_peak = p.do_profile && !skipped;
      if (p.ev.peak) p.ev.peak[e] = have_peak ? peak : -1;
      if (p.ev.flow) p.ev.flow[e] = flow;
      if (p.ev.job_steps) p.ev.job_steps[e] = steps;
      if (p.ev.horizon) p.ev.horizon[e] = hmax;
      if (p.ev.n_unfinished) p.ev.n_unfinished[e] = unfinished;
      if (p.ev.feasible) p.ev.feasible[e] = (have_peak && !(status & KVS_EVAL_RANGE) && peak <= M) ? 1 : 0;
      if (p.ev.status) p.ev.status[e] = status;
      if (p.out.n_runs) p.out.n_runs[e] = sh.n_runs;
    }
    (void)want32;
  }
}

}  // namespace

static size_t fused_smem_bytes(bool light) { return light ? offsetof(FShared, dA) : sizeof(FShared); }

template <bool LIGHT, int FAM, bool VARIANTS>
static int ctas_per_sm() {
  int n = 0;
  cudaFuncSetAttribute(k_fused_eval<LIGHT, FAM, VARIANTS>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(fused_smem_bytes(LIGHT)));
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_fused_eval<LIGHT, FAM, VARIANTS>, KVS_EVAL_THREADS, fused_smem_bytes(LIGHT)) != cudaSuccess) n = 1;
  return n < 1 ? 1 : n;
}

// CTAs per SM that every instantiation used for this kind of launch reaches.
int kvs_fused_ctas_per_sm(int light) {
  int n;
  if (light) {
    n = ctas_per_sm<true, KVS_FUSED_ANY, true>();
    n = min(n, min(min(ctas_per_sm<true, KVS_GBA, true>(), ctas_per_sm<true, KVS_GSA, true>()), min(ctas_per_sm<true, KVS_SPS, true>(), ctas_per_sm<true, KVS_SIMS, true>())));
  } else {
    n = min(ctas_per_sm<false, KVS_FUSED_ANY, true>(), min(ctas_per_sm<false, KVS_GBA, false>(), ctas_per_sm<false, KVS_GSA, true>()));
    n = min(n, min(min(ctas_per_sm<false, KVS_FUSED_SHARED, false>(), ctas_per_sm<false, KVS_FUSED_SHARED, true>()), ctas_per_sm<false, KVS_FUSED_SHARED_EST, false>()));
  }
  return n;
}

template <bool LIGHT, int FAM, bool VARIANTS>
static cudaError_t launch(const BuildParams& p, int grid, cudaStream_t stream) {
  k_fused_eval<LIGHT, FAM, VARIANTS><<<grid, KVS_EVAL_THREADS, fused_smem_bytes(LIGHT), stream>>>(p);
  return cudaGetLastError();
}

// The caller zeroes the counters; kvs_fused_ctas_per_sm has set the kernels up.  light: the variant without the ring (see k_fused_eval); fam:
// KVS_FUSED_ANY, KVS_FUSED_SHARED where p.parts > 1, or a family id for a list of that family alone in a call without estimates (the
// full variant has such kernels for the two geometric families, the light one for all four).
cudaError_t kvs_launch_fused(const BuildParams& p, int grid, int light, int fam, cudaStream_t stream) {
  if (p.P <= 0) return cudaSuccess;
  if (light) {
    switch (fam) {
      case KVS_GBA: return launch<true, KVS_GBA, true>(p, grid, stream);
      case KVS_GSA: return launch<true, KVS_GSA, true>(p, grid, stream);
      case KVS_SPS: return launch<true, KVS_SPS, true>(p, grid, stream);
      case KVS_SIMS: return launch<true, KVS_SIMS, true>(p, grid, stream);
      default: return launch<true, KVS_FUSED_ANY, true>(p, grid, stream);
    }
  }
  if (fam == KVS_GBA) return launch<false, KVS_GBA, false>(p, grid, stream);
  if (fam == KVS_GSA) return launch<false, KVS_GSA, true>(p, grid, stream);
  if (fam == KVS_FUSED_SHARED && p.key) return launch<false, KVS_FUSED_SHARED_EST, false>(p, grid, stream);
  if (fam == KVS_FUSED_SHARED) return p.variants ? launch<false, KVS_FUSED_SHARED, true>(p, grid, stream) : launch<false, KVS_FUSED_SHARED, false>(p, grid, stream);
  return launch<false, KVS_FUSED_ANY, true>(p, grid, stream);
}

// First violation recorded by the checked build (0 = none); `compiled` = 1 if this library was built with
// -DKVS_DEBUG.  `reset` clears the word after reading it.
cudaError_t kvs_fused_check_word(unsigned long long* word, int* compiled, int reset) {
#ifdef KVS_DEBUG
  if (compiled) *compiled = 1;
  cudaError_t e = cudaMemcpyFromSymbol(word, g_check_word, sizeof(unsigned long long));
  if (e == cudaSuccess && reset) { const unsigned long long z = 0ull; e = cudaMemcpyToSymbol(g_check_word, &z, sizeof(z)); }
  return e;
#else
  if (compiled) *compiled = 0;
  *word = 0ull;
  (void)reset;
  return cudaSuccess;
#endif
}
