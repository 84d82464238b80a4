// Calls of csrc/lmhead.cu on the stand-in runtime of fake_launch_limits.cpp.
#include "../paper_2402_11809_b200/csrc/common.cuh"

void fake_limits_reset(int at, int (*other)());
size_t fake_largest_launch();

namespace {
const space_lmhead_args* other_args;
int other_rc;

int call(const space_lmhead_args* a, int* launches = nullptr) {
  static char scratch[64];                        // (never read or written: nothing runs)
  space_ctx* c = new space_ctx();
  c->sm_count = 148;
  c->lm_part = c->lm_gather = scratch;
  c->lm_counter = reinterpret_cast<int*>(scratch);
  const int rc = launch_lmhead_verify(c, a, nullptr);
  if (launches) *launches = (int)c->launches;
  delete c;
  return rc;
}
int other_call() { return other_rc = call(other_args); }
}  // namespace

// One call of `a`; before its launch number `at`, a whole call of `b` on another context.  Results in rc[0], rc[1], the
// dynamic shared memory of the largest launch in *smem.
extern "C" void fake_lmhead_two(const space_lmhead_args* a, const space_lmhead_args* b, int at, int* rc, size_t* smem) {
  other_args = b; other_rc = SPACE_OK;
  fake_limits_reset(at, other_call);
  rc[0] = call(a);
  rc[1] = other_rc;
  *smem = fake_largest_launch();
}

// Launches that a call of `a` takes.
extern "C" int fake_lmhead_launches(const space_lmhead_args* a) {
  int n = 0;
  fake_limits_reset(0, nullptr);
  return call(a, &n) == SPACE_OK ? n : -1;
}
