// How the speculative runs' kernel with its state in shared memory (k_spec_smem in kvs_spec.cu) is laid out and launched: bytes of a CTA, and
// how many evaluations of one instance a CTA takes.  Host code, but for the sizes, which the kernel uses too.
#pragma once

#include <algorithm>
#include <vector>

#include "kvs_internal.cuh"

#ifdef __CUDACC__
#define KVS_BOTH __host__ __device__
#else
#define KVS_BOTH
#endif

constexpr int SPEC_WARPS = KVS_SPEC_GROUP;   // evaluations of one CTA, at most
constexpr int SPEC_SM_WARPS = 16;            // of one SM: what the kernel's 115 registers allow
constexpr int RING_MAX = 1024, RING_MIN = 256;
constexpr int STK_BLK = 64;
constexpr int SPEC_TABLE_BYTES = 4 * 4 * KVS_MAX_PHASES + 4 * (KVS_MAX_PHASES + 1) + 4 + 2 * 8 + 8;
constexpr int SPEC_POWERS_BYTES = 2 * 16 * (KVS_MAX_PHASES + 1);
constexpr int SPEC_SMEM = 227 * 1024;        // of one CTA
constexpr int SPEC_SM_SMEM = 228 * 1024;     // of one SM, 1 KB of it taken by each CTA besides its own

// Bytes of one warp's state for instances of at most n jobs with a ring of that many rounds, and of the lengths that a CTA's warps share.
KVS_BOTH inline int smem_jobs(int n) { return (n + 127) & ~127; }
KVS_BOTH inline int smem_stack_bytes(int m) { return 2 * m > SPEC_POWERS_BYTES ? 2 * m : SPEC_POWERS_BYTES; }
KVS_BOTH inline int smem_state_bytes(int n, int ring) {
  const int m = smem_jobs(n);
  return SPEC_TABLE_BYTES + ring * 8 + smem_stack_bytes(m) + 2 * m + 2 * (m / 8) + ((m / STK_BLK * 4 + 15) & ~15);
}
KVS_BOTH inline int smem_lengths_bytes(int n) { return smem_jobs(n) * 4; }

inline int spec_cta_bytes(int n, int warps, int ring) { return smem_lengths_bytes(n) + warps * smem_state_bytes(n, ring); }
// CTAs that an SM holds; 0: not one.
inline int spec_resident(int n, int warps, int ring) {
  const int bytes = spec_cta_bytes(n, warps, ring);
  return bytes > SPEC_SMEM ? 0 : std::min(SPEC_SM_SMEM / (bytes + 1024), SPEC_SM_WARPS / warps);
}

// Bytes of scratch of a CTA: a 16-bit list of participants per evaluation.
inline i64 spec_list_bytes(i64 max_jobs, int warps) { return 2ll * warps * ((max_jobs + 127) & ~127ll); }

// Evaluations per CTA and rounds of the ring for a call; warps = 0: the kernel in global memory takes all of them.
struct SpecShape { int warps = 0, ring = 0; i64 groups = 0; };

// Groups that an instance's evaluations are cut into, of sizes that differ by one at most.
inline i64 spec_groups(i64 evals, int warps) { return (evals + warps - 1) / warps; }

// A launch has one width, so a CTA is made as wide as leaves the most evaluations in flight: its warps share the instance's lengths, but
// what a smaller group leaves empty is lost, and so is what does not make a whole CTA on an SM.  Where several widths have all
// evaluations in flight, the widest (512 evaluations of 5,000 jobs, eight budgets: 10.5 ms, 10.9 one per CTA); where equally many have
// to take turns, the narrowest, whose places become free one by one (8,192 of 10,000 jobs, two budgets: 331 ms one per CTA, 355
// two; of 500 jobs 13.6 and 15.3).  A ring of 1,024 rounds is given up only where a shorter one lets in another CTA.
//
// An SM then has `live` of its evaluations in flight and takes evaluations / live chains for them.  The kernel in memory, 32 slower chains
// per SM, takes as long as 13.5 of these for a few evaluations and a fifth of one more for each.  ms on chip / in memory, config 2's lengths:
//   24,000 jobs, one budget per instance (1 live): 90 / 272 (512 evaluations), 336 / 365 (2,048), about 500 / 402 (3,072);
//   16,000 jobs, one (1): 64 / 204, 237 / 267 (2,048), 282 / 274 (2,400), 932 / 514 (8,192);
//   five (1.67): 47 / 201, 165 / 254, 628 / 520 (8,192);  two (2): 44 / 201, 144 / 264, 416 / 383 (6,000), 562 / 516 (8,192);
//   10,000 jobs, one (2): 24 / 130, 85 / 178, 244 / 245 (6,000), 331 / 338 (8,192);  five (2.5): 24 / 146, 79 / 164, 298 / 339 (8,192);
//   eight (4): 18 / 135, 61 / 165, 219 / 395 (8,192);
//   5,000 jobs, one (4): 11 / 91, 30 / 111, 108 / 185 (8,192);  500 jobs, one (16): 3.2 / 23, 4.7 / 25, 13.5 / 34 (8,192).
// (With room for four evaluations in every CTA, one budget per instance: 48, 174, 683 ms at 10,000 jobs, 27, 97, 380 at 5,000, 31 at 500 and 8,192.)
inline SpecShape kvs_spec_shape(i64 max_jobs, const std::vector<i64>& evals_of, int sm_count) {
  SpecShape best;
  if (max_jobs >= 65535) return best;        // 16-bit job numbers, one of them spare
  const int n = static_cast<int>(max_jobs);
  i64 evals = 0, narrower = 0;
  for (i64 c : evals_of) evals += c;
  double best_share = 0.0;                   // of the evaluations that are in flight at a time
  for (int w = 1; w <= SPEC_WARPS; ++w) {
    SpecShape x;
    x.warps = w;
    for (i64 c : evals_of) x.groups += spec_groups(c, w);
    if (x.groups == narrower) continue;      // no group has w of them
    narrower = x.groups;
    double share = 0.0;
    for (int ring = RING_MAX; ring >= RING_MIN; ring /= 2) {
      const i64 held = static_cast<i64>(spec_resident(n, w, ring)) * sm_count;
      const double y = held < x.groups ? static_cast<double>(held) / static_cast<double>(x.groups) : 1.0;
      if (y > share) { share = y; x.ring = ring; }
    }
    if (share > best_share || share == 1.0) { best_share = share; best = x; }
  }
  const double per_sm = static_cast<double>(evals) / sm_count;
  if (best_share < 1.0 && 1.0 / best_share > 13.5 + per_sm / 5.0) return SpecShape{};   // per_sm / live chains on chip
  return best;
}
