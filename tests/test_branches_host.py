"""The branch streams and events of the captured per-instance sweep: when a
creation fails, the next call makes what is missing (host stand-ins of the
CUDA calls; every creation in turn fails)."""
from __future__ import annotations

from tests import cpp_extract

_PROGRAM = """
#include <cstdio>
enum { QISG_OK = 0, QISG_ECUDA = -3 };
typedef int *cudaStream_t;
typedef int *cudaEvent_t;
enum { cudaStreamNonBlocking, cudaEventDisableTiming };
static int made = 0, fail_at = 0;
static int pool[64];
static int make(int **p) {
  if (fail_at && ++made == fail_at) return 1;
  static int n = 0;
  *p = &pool[n++ %% 64];
  return 0;
}
static int cudaStreamCreateWithFlags(cudaStream_t *s, int) { return make(s); }
static int cudaEventCreateWithFlags(cudaEvent_t *e, int) { return make(e); }
static int cuda_check(int e, const char *) { return e ? QISG_ECUDA : QISG_OK; }
constexpr int kLanesBranches = 8;
struct qisg_handle {
  cudaStream_t branch[kLanesBranches] = {};
  cudaEvent_t fork_ev = nullptr, join_ev[kLanesBranches] = {};
};
%s
int main() {
  for (int k = 1; k <= 2 * kLanesBranches + 1; ++k) {
    qisg_handle h;
    made = 0;
    fail_at = k;
    if (lanes_make_branches(&h) != QISG_ECUDA) return 1;
    fail_at = 0;
    if (lanes_make_branches(&h)) return 2;
    if (!h.fork_ev) return 3;
    for (int b = 0; b < kLanesBranches; ++b)
      if (!h.branch[b] || !h.join_ev[b]) return 4;
    const cudaEvent_t kept = h.fork_ev;
    if (lanes_make_branches(&h) || h.fork_ev != kept) return 5;
  }
  std::printf("ok");
}
"""


def test_a_failed_creation_is_made_up_for(tmp_path):
    body = cpp_extract.function("lanes.cu", "int lanes_make_branches(")
    assert cpp_extract.run(tmp_path, _PROGRAM % body) == "ok"
