// Which form of the neighbourhood search and of the small-neighbourhood LP
// (n = 1) a step takes: by the capacity where the schedule leaves it to the
// step, else the one that the schedule names.
#pragma once

namespace vrm {

// What every context starts with.  These values leave the form to the step;
// any other one is the caller's choice and holds at every capacity.  (A rule on
// the values and not on whether a schedule was set: an answer of
// vrm_get_schedule set again, with another field changed or not, changes no
// form.)
constexpr int kSearchBlockDefault = 256, kLpBlockDefault = 128, kLpBlocksPerSmDefault = 16;

constexpr int kLpWsThreads = 192;      // lp_block of the 4 + 2-warp form
constexpr int kLpWsThreadsWide = 384;  // lp_block of the 8 + 4-warp form

// Largest capacity (of all clouds that run at the same time) whose cell scans
// give a warp to each particle or proposal instead of a thread: at 870
// particles a thread's chain of dependent loads over nine cells takes 33 us in
// the neighbourhood search and in the masks (7 and 9 by warps), 17 in the mask
// update (10) and 8 in the conflict test (5); at 20,449 34, 14, 21 and 11
// against 20, 11, 21 and 7.
constexpr int kWarpScanCap = 65536;

// Largest particle capacities whose n = 1 LPs all go to the pairs kernel, eight
// lanes per LP, and whose hand-backs do.  One LP per thread takes 32 us in
// binary32 and 43 for the re-run of a few in FP64 however few they are, the
// pairs and their solves 35 for all; but they take seven times the
// instructions.  Steps of 3,600, 20,449 and 32,400 particles: 290, 323 and 386
// us with all LPs in pairs, 346, 371 and 409 with binary32 and FP64 (65,536:
// 435 and 446, 90,000: 511 and 483).  Hand-backs in pairs: 423, 474, 509 and
// 578 us at 65,536, 90,000, 129,600 and 184,900 particles against 446, 483,
// 531 and 582, but 1,675 against 1,664 at a million.  The capacity is what the
// host knows; twice the particles is usual.  The clouds of a batch run at the
// same time, so the sum of their capacities counts there (32 clouds of 10,000
// to 300,000 particles: 4.49 ms, 4.60 when each went by its own).
constexpr int kPairsCap = 65536;
constexpr int kPairsRetryCap = 6 * 65536;
// Smallest capacity that takes the 8 + 4-warp form: steps of 640,000 particles
// 1,075 us against 1,114 with one kind of warp, of a million 1,469 against
// 1,581; 787 and 797 at 360,000.  The form fills every SM, so batches, whose
// clouds run beside each other, keep the other (4.54 ms against 4.66), as do
// capacities that may hold fewer LPs than this (an RK3 step of 500,000 in
// 730,000: 2.41 against 2.47 ms).
constexpr int kWsCap = 18 * 65536;

enum LpForm { kLpPairs, kLpThreads, kLpWs, kLpWsWide };

// cap: this cloud's capacity; load: that of all clouds running at the same time
// in a batch, 0 for a cloud by itself.
inline LpForm small_lp_form(int lp_block, int lp_blocks_per_sm, int cap, int load) {
  if (lp_block == kLpWsThreads) return kLpWs;
  if (lp_block == kLpWsThreadsWide) return kLpWsWide;
  if (lp_block != kLpBlockDefault || lp_blocks_per_sm != kLpBlocksPerSmDefault) return kLpThreads;
  if ((load > cap ? load : cap) <= kPairsCap) return kLpPairs;
  return load == 0 && cap >= kWsCap ? kLpWsWide : kLpThreads;
}

// The step's neighbourhood search with a warp per particle (small clouds).
inline bool search_by_warps(int search_block, int cap, int load) {
  return search_block == kSearchBlockDefault && (load > cap ? load : cap) <= kWarpScanCap;
}

}  // namespace vrm
