// Bit-matrix fixpoint of chain programs under the unit semiring (bitmat.cu).
#pragma once
#include "kernels.h"

struct lob_engine;

// Plans the run; false when the program is not a chain program or an option
// asks for another strategy.  Needs the column widths and idb flags.
bool bit_eligible(const lob_engine& e);
// Runs the loaded program to its fixpoint on bit matrices.  Returns false, with
// nothing allocated, when the domain is too large, the facts are likely to be few for
// it (e.bit_watch is set then) or memory runs out (the general path then runs); else
// *rc is LOB_OK or LOB_E_MAXITER, and the relations' sizes, k and the statistics are
// set.
bool bit_run(lob_engine& e, u32 max_iters, u32& k, u64& new_facts, int* rc);
// While e.bit_watch is set: the iteration to come is likely to derive so much that the
// run had better start again on bit matrices (join fan-outs as for facts spread evenly).
bool bit_blow_up(const lob_engine& e);
// Rows of a derived relation, read out of its bit matrix (unit tags).
void bit_read(lob_engine& e, u32 rel, u32* cols, u64 stride, float* tags, u32* samples);
// Gives the matrices back.
void bit_release(lob_engine& e);
