// The shared scan by table lookup (esc_boxes.cu), as the entry points of
// esc_scan.cu use it.
#pragma once
#include <cuda_runtime.h>

#include "esc_internal.h"
#include "esc_stage.h"

namespace esc {

constexpr int kMaxBoxes = 16;          // disjoint boxes of one predicate
constexpr int kMaxPassBoxes = 8192;    // boxes of one pass
constexpr int kMaxOperands = 24;       // distinct operands of one pass
constexpr int kMaxUdfOperands = 8;     // udfs among them
constexpr uint64_t kMaxTableBytes = (uint64_t)64 << 20;
constexpr int kMaxBoxSmem = 220 * 1024;

// One test of a predicate, on the value of one operand.
struct BoxTest {
  int64_t lo, hi;      // OP_RANGE: inclusive bounds
  uint32_t operand;
  uint32_t off;        // OP_IN, OP_INSET: first entry in the pass's pool
  uint16_t n;          // OP_IN, OP_INSET: values
  uint8_t op;
  uint8_t pad[5];
};
static_assert(sizeof(BoxTest) == 32, "BoxTest layout");

struct BoxPlan;
enum BoxFit { BOX_ADDED, BOX_FULL, BOX_NEVER };
BoxPlan *new_box_plan();
void free_box_plan(BoxPlan *p);
// Adds a predicate's boxes; their counts go to counts[index].  BOX_FULL: it
// does not fit beside those already there; BOX_NEVER: not even alone.
BoxFit add_predicate(BoxPlan *plan, const esc_pred *p, uint32_t index);
// Enqueues the pass.  *done is false, and nothing is enqueued, when its table
// would be too large or no predicate reads a column.
esc_status run_boxes(BoxPlan *plan, const esc_table *t, int sms, unsigned long long *counts, ScratchHdr *hdr,
                     cudaStream_t st, bool *done);

// Device memory that a pass over at most n predicates allocates, at most.
uint64_t box_scratch_bound(uint64_t n);

// Stream-ordered allocation from the library's device pool (esc_scan.cu).
esc_status alloc_async(void **p, size_t bytes, cudaStream_t st);

}  // namespace esc
