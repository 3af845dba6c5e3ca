// ragged.cuh -- the grouped form of a ragged batch's divisions and products
// (ragged.cu): host-side plan and launch.
#pragma once
#include <cstdint>
#include <vector>

#include "common.cuh"

namespace bigint {

// One operation of the grouped form: u / v (or the product of the operands u
// and v), limb offsets into the input pool, of the results into the output
// pool, and of the operation's records from the base of its wave's.
struct RagOp {
  int32_t nu, nv;
  int32_t opi;  // operation index (status)
  int32_t pad;
  int64_t u, v, q, r, rec;
};

// Product forms of a grouped launch (tc_choose).
enum RagShape {
  RAG_ONE128, RAG_ONE256, RAG_64, RAG_128, RAG_256, RAG_PIPE128, RAG_PIPE64,
  RAG_PIPE128N, RAG_PIPE64N,  // with 128-column tiles
  RAG_NSHAPES
};

// A list of operations (RagOp indices, RAG_SWAP set where the second operand
// is the one stored whole in shared memory) whose products of one kind run
// in one launch.
constexpr int32_t RAG_SWAP = 1 << 30;
enum RagKind { RAG_P, RAG_P2, RAG_UW, RAG_QV, RAG_MUL };

// One launch of the program.
enum RagWhat { RAG_START, RAG_SMALL, RAG_PROD, RAG_MID, RAG_UPDATE, RAG_FINISH };
struct RagLaunch {
  int what, kind, l, par;  // step (limbs known before it), parity of its iterate
  bool sibling;            // RAG_PROD: independent of the launch before it
  int shape, grid;
  uint32_t smem;           // RAG_PROD: dynamic shared memory
  int nx;                  // largest operand stored whole
  int64_t first, n;        // RAG_PROD: range of the list; else ops [first, first + n)
};

struct RagPlan {
  std::vector<RagOp> ops;       // waves of divisions one after the other, then products
  std::vector<int32_t> list;
  std::vector<RagLaunch> program;
  int64_t ndiv = 0;
  size_t rec_bytes = 0;         // largest wave's records
};

// Whether every product of a division of nu by nv limbs (mul: the product
// itself) has a form: an operand of each has to lie in shared memory whole,
// which a quotient of some 11000 limbs and more is too long for.
bool rag_takes(int nu, int nv, bool mul);

// Plans the given operations (divisions with nv >= 8 and nu >= nv, products,
// all of which rag_takes); BIGINT_OK or BIGINT_ECUDA.
int rag_plan(std::vector<RagOp> divs, std::vector<RagOp> muls, RagPlan &P);

// Device buffers of a launch: plan copies, records, the irregular divisions'
// list (operation indices, ndiv entries) and two counters (irregular count,
// a product gave up), zeroed here.
struct RagBuffers {
  const RagOp *ops;
  const int32_t *list;
  uint64_t *rec;
  int32_t *irregular;
  int *ctr;
};
int rag_launch(const RagPlan &P, const RagBuffers &B, const uint64_t *in, uint64_t *out,
               int32_t *status, cudaStream_t st);

}  // namespace bigint
