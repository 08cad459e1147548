// Test harness: the packed-stream plan of the preconditioner apply (csrc/setup.cpp,
// build_stream) for the CPU tests. Built by tests/test_stream_plan.py with the
// host compiler.
#include <string>
#include <vector>

#include "setup.h"

using namespace fsi;

struct Box {
  RasPlan R;
  StreamPlan S;
};

extern "C" void* stream_new(int64_t n, const double* X, int64_t T, const int32_t* tets, int32_t np, int32_t fill,
                            int32_t ordering, const uint8_t* rank, int64_t cut, int64_t most, int64_t stage) {
  auto* b = new Box;
  std::vector<int32_t> tv(tets, tets + 4 * T);
  b->R = build_ras(build_pattern(n, tv), X, n, nullptr, 1, np, 1, fill, ordering, rank);
  b->S = most > 0 ? build_stream(b->R, cut, most, stage) : build_lookahead_stream(b->R, stage);
  return b;
}

extern "C" void stream_free(void* p) { delete static_cast<Box*>(p); }

extern "C" const void* stream_array(void* p, const char* name, int64_t* count) {
  Box& B = *static_cast<Box*>(p);
  const std::string s(name);
#define ARR(owner, field)                    \
  if (s == #field) {                         \
    *count = (int64_t)B.owner.field.size();  \
    return B.owner.field.data();             \
  }
  ARR(R, sd_row) ARR(R, row_ptr) ARR(R, col) ARR(R, diag)
  ARR(S, L_off) ARR(S, U_off) ARR(S, src) ARR(S, piv) ARR(S, code) ARR(S, code_off)
  ARR(S, stage_off)
#undef ARR
  if (s == "bcol") {
    *count = (int64_t)B.S.col.size();
    return B.S.col.data();
  }
  if (s == "stage") {
    *count = (int64_t)B.S.stage.size();
    return B.S.stage.data();
  }
  *count = -1;
  return nullptr;
}
