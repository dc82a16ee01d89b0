// Linear recursion of tagged programs in one launch (linear.cu).
#pragma once
#include <utility>
#include <vector>

#include "common.cuh"

struct lob_engine;
struct lob_stats;

// What the linear components of a run left behind: their relations, the
// iteration they stopped in, whether max_iters stopped them, and per iteration
// from `first` on each relation's (|F|, |recent|) at its start.
struct LinearOut {
  bool taken = false, max_iter = false;
  u32 first = 2, last = 1;
  std::vector<u32> rels;
  // [iteration - first][index in rels]; kept up only where a backward pass
  // reads it (the add-mult semirings)
  std::vector<std::vector<std::pair<u64, u64>>> counts;
  std::vector<u64> n_recent;                             // after the last iteration
};
// Runs every linear component of the program from iteration 2 to its fixpoint
// (or max_iters).  Its relations then have no recent facts; the caller runs the
// rest of the program and merges the counts (linear_merge).
void run_linear(lob_engine& e, u32 max_iters, lob_stats& s, LinearOut& out);
// The whole run ended in iteration k: writes the components' counts into the
// engine's per-iteration record.
void linear_merge(lob_engine& e, u32 k, const LinearOut& out);

// top-1-proofs: the run's proof arena, and what follows kernels that append to it
// (engine.cu)
struct Top1Arena;
Top1Arena top1_desc(lob_engine& e);
bool top1_settle(lob_engine& e);

// diff-add-mult backward of the linear components' iterations after the first.
// Device pointers by relation id: adjoints and dense key -> row maps (null: none),
// and per view its rows' primary rows.  needed: relations that carry adjoints; a
// component with none of them is left out.  Flags the components' relations; false
// when there is none to take (the caller replays every iteration).  extra is set
// once memory is asked for.
struct LinearAdjoints {
  std::vector<double*> adj;
  std::vector<u32*> hrow;
  std::vector<std::vector<u32*>> prow;
};
bool linear_backward(lob_engine& e, const LinearAdjoints& J, const std::vector<char>& needed, std::vector<char>& in,
                     bool& extra);
