"""The batched LUs' helper streams after a launch that fails: whatever was launched on them is joined
back into the caller's stream, so that what the caller does next on it comes after their kernels. On
the CPU, from the launcher's source with stand-ins for the CUDA calls."""
import pytest

import cuda_on_host


@pytest.mark.parametrize("good", [0, 1, 3, 14, 99])  # launches before the one that fails
def test_helper_streams_are_joined(tmp_path, good):
    cuda_on_host.run(tmp_path, [], r"""
typedef int cudaStream_t;
typedef int cudaEvent_t;
static constexpr int32_t cudaSuccess = 0, RLU_OK = 0, RLU_EINVAL = 1, RLU_ECUDA = 4;
static constexpr int kLuGroups = 19, kLuSide = 12, kLuNarrow = 48;
struct LuArgs {};
struct LuFork { cudaStream_t hs[kLuSide]; cudaEvent_t fork, join[kLuSide]; };
#define RLU_CUDA_TRY(e) do { if ((e) != 0) return RLU_ECUDA; } while (0)
#define RLU_TRY(e) do { int32_t s_ = (e); if (s_ != RLU_OK) return s_; } while (0)
static int launched = 0;
static bool forked[100], pending[100];   // by stream: waits for the fork; holds unjoined work
static int recorded_on[100];             // by event: the stream it was last recorded on
static int cudaEventRecord(cudaEvent_t e, cudaStream_t s) { recorded_on[e] = s; return 0; }
static int cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, int) {
  if (s == 0) pending[recorded_on[e]] = false;
  else forked[s] = true;
  return 0;
}
template <int RT>
static int32_t lu_batched_group(bool, const LuArgs*, int, int, int, int, cudaStream_t s) {
  CHECK(s == 0 || forked[s]);
  if (launched++ == GOOD) return RLU_ECUDA;
  pending[s] = s != 0;
  return RLU_OK;
}
""".replace("GOOD", str(good)) + cuda_on_host.definition("lu_reg.cu", "launch_lu_reg_batched") + r"""
int main() {
  LuFork f;
  f.fork = 0;
  for (int i = 0; i < kLuSide; ++i) {
    f.hs[i] = 1 + i;
    f.join[i] = 1 + i;
  }
  int first[kLuGroups] = {}, count[kLuGroups] = {}, wide[kLuGroups] = {};
  int parts = 0;
  for (int g = 1; g < kLuGroups; ++g) {
    count[g] = 2;
    wide[g] = g < 12 ? 1 : 2;  // some groups in two parts: 29 launches
    parts += g < 12 ? 2 : 1;
  }
  const int32_t st = launch_lu_reg_batched(false, 512, nullptr, first, count, wide, 0, &f);
  CHECK(st == (launched <= GOOD ? RLU_OK : RLU_ECUDA));
  CHECK(launched == (GOOD < parts ? GOOD + 1 : parts));
  for (int i = 0; i < 100; ++i) CHECK(!pending[i]);
}
""".replace("GOOD", str(good)))
