// team.h -- what the team pass (team.cuh) shares with its host driver.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include "internal.h"

namespace lk {

enum { TEAM_BLOCK = 0, TEAM_CLUSTER = 1, TEAM_GRID = 2 };
// How a team pass ended: globally converged after the refinement; renumbered
// to as many communities as vertices (aggregation would not shrink the
// graph); renumbered only (the caller aggregates); aggregated; nothing done,
// the level's hubs exceed the scratch.
enum { TEAM_NONE = 0, TEAM_CONVERGED = 1, TEAM_NO_SHRINK = 2, TEAM_RENUMBERED = 3, TEAM_AGGREGATED = 4, TEAM_TOO_BIG = 5 };

// Distinct candidates of a vertex the block's table takes (half its slots);
// vertices with more are hubs.  Hubs of a colour class whose eligibility a
// block notes once a sub-sweep.
static constexpr int64_t TEAM_MAX_CAND = 8192;
static constexpr int TEAM_MAX_HUBS = 16384;
static constexpr int TEAM_MAX_BLOCKS = 1024;
// Polls of a grid barrier before it gives up (the default takes several seconds).
#ifndef LK_TEAM_SPIN_LIMIT
#define LK_TEAM_SPIN_LIMIT (1ull << 24)
#endif
static constexpr u64 TEAM_SPIN_LIMIT = LK_TEAM_SPIN_LIMIT;

// Control words of a team, zeroed before every pass.
struct TeamCtl {
  unsigned bar, abort;
  unsigned npiece[2];      // row pieces the whole team re-marks, by parity
  unsigned nover[2];       // proposals beyond the blocks' own lists, by parity of the sub-sweep
  u64 sums[2][2];          // sum of S of the current / next iteration (i128)
  u64 scanned_e, scanned_v, cand, changed, rmoves;
  int64_t moves;
  int32_t li, status, too_big, pad0;
  int64_t nc, nnz2;
  u64 maxdeg, kmax;        // of the aggregated level
  u64 decide_ns, subsweeps;
  u64 stamp[4];            // globaltimer at the start and after local-moving, refinement, aggregation (or renumbering)
  // end of the part the host reads back
  int64_t part[TEAM_MAX_BLOCKS];
  unsigned ktot[256 * 8], kcur[256 * 8];
};
static constexpr size_t TEAM_CTL_HEAD = offsetof(TeamCtl, part);

// Arrays of the current level; n and nnz bound them all.
struct TeamArrays {
  // A class with more hubs than a block notes makes the pass give up
  // (TEAM_TOO_BIG; the context runs it on the multi-kernel path).  Where there
  // is no other path, the hubs beyond are asked again per item, which cost
  // hub-heavy passes of a context 1% (Chung-Lu DF) for code they hardly reach.
  static constexpr bool MANY_HUBS = false;
  int32_t *C, *CB, *rep, *vlist;
  int64_t *K, *Sig, *Sig2;
  uint8_t *ch, *ch2, *processed, *stamp, *exists;
  int32_t *prop_i, *prop_c;
  u64 *err;
  // hubs: table scratch (tcap slots, empty whenever nobody uses it), prefix
  // sums of insert and scan items, finished scan items and their results
  int32_t *tkeys;
  u64 *tvals;
  int64_t tcap;
  int32_t *hub_i, *hub_s, *hub_done, *part_c;
  i128 *part_sc;
  int64_t *part_kid;
  // long rows to re-mark: mover and piece (at most 2 * nnz / REMARK_PIECE)
  int32_t *piece_i, *piece_k;
  // aggregation: table keys and sums, row entry counts and cursors, row sums,
  // and the output graph
  u64 *hkey, *hval;
  int64_t *cnt, *cur, *K2;
  int64_t *off2;
  int32_t *idx2;
  int64_t *w2;
};

// One pass on a level graph of WT weights with scores of ST.  Reads the level
// (off, idx, w), K', Sigma', C', processed, changed flags (and the DS range);
// leaves the renumbered C' also in CB for the dendrogram lookup and, when it
// aggregates (agg_slots > 0), the next level's graph and its initial state.
// Sig / Sig2 and ch / ch2 have changed places when it returns.
template <typename WT>
struct TeamArgs {
  GraphView<WT> g;
  int64_t nnz;
  TeamArrays a;
  int64_t A, p, two_m;
  double den, tau;
  int log2S, dynamic, timing, lp, max_iters;
  int64_t agg_slots;       // aggregation table (0: the caller aggregates)
  const uint8_t *in_range;
  TeamCtl *ctl;
};
// Launches the pass over nb blocks (one per SM at most) as `kind`; an error
// when the runtime refuses the launch (nothing is enqueued then).
static constexpr int TEAM_MAX_CLUSTER = 16;
template <typename WT, typename ST>
bool team_cluster_fits(int nb);
template <typename WT, typename ST>
int launch_team_pass(const TeamArgs<WT> &args, int nb, int kind, cudaStream_t s);

}  // namespace lk
