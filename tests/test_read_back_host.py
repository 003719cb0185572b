"""qisg_overlaps on host stand-ins of the CUDA calls: the counts are cleared
before the call's synchronisation, whatever the device's error flag says."""
from __future__ import annotations

import pytest

from tests import cpp_extract

_PROGRAM = """
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <string>
enum { QISG_OK = 0, QISG_EINVAL = -1, QISG_ECUDA = -3, QISG_ETIMEOUT = -4 };
enum { QISG_LAYOUT_LANES = 1, QISG_LAYOUT_SAMPLES = 2, QISG_LAYOUT_SITES = 3 };
typedef void *cudaStream_t;
typedef int cudaError_t;
enum { cudaMemcpyDeviceToHost };
static std::string log_;
static int cudaMemcpyAsync(void *d, const void *s, size_t n, int, cudaStream_t) { std::memcpy(d, s, n); log_ += 'c'; return 0; }
static int cudaMemcpy(void *d, const void *s, size_t n, int) { std::memcpy(d, s, n); log_ += 'C'; return 0; }
static int cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); log_ += 'm'; return 0; }
static int cudaStreamSynchronize(cudaStream_t) { log_ += 's'; return 0; }
struct qisg_handle {
  cudaStream_t stream = nullptr;
  unsigned char *pin = nullptr;
  int *d_err = nullptr;
  long long *d_q = nullptr;
  int layout = QISG_LAYOUT_SAMPLES;
  int64_t n_samples = 1, n_a_pad = 2, n_slots = 1;
  int n_pairs() const { return 1; }
};
static int fail(int code, const char *) { return code; }
static int cuda_check(cudaError_t e, const char *) { return e; }
static int lanes_measure(qisg_handle *, int) { return 0; }
static int sites_measure(qisg_handle *, int) { return 0; }
static int samples_measure(qisg_handle *h, int) { h->d_q[0] = 17; return 0; }
constexpr size_t kPinBytes = 256 << 10;
%s;
%s
%s
%s
int main() {
  static unsigned char pin[kPinBytes];
  long long q[2] = {0, 0};
  int err = %d;
  qisg_handle h;
  h.pin = %d ? pin : nullptr;
  h.d_err = &err;
  h.d_q = q;
  int64_t out = 0;
  const int rc = qisg_overlaps(&h, &out);
  std::printf("%%d %%d %%d %%d", rc, (int)out, (int)q[0], log_.find_last_of("m") < log_.find('s'));
}
"""


@pytest.mark.parametrize("pinned", [0, 1])
@pytest.mark.parametrize("err,rc,q", [(0, 0, 17), (1, -4, 17)])
def test_overlaps_clear_their_counts(tmp_path, pinned, err, rc, q):
    api = "qisg_api.cu"
    parts = (cpp_extract.function("qisg_internal.cuh", "struct ReadBack"),
             cpp_extract.function(api, "int read_back(cudaStream_t st,"), cpp_extract.function(api, "int read_back(qisg_handle *h,"),
             cpp_extract.function(api, "int qisg_overlaps("))
    got = [int(x) for x in cpp_extract.run(tmp_path, _PROGRAM % (*parts, err, pinned)).split()]
    assert got[0] == rc and got[2] == 0 and got[3] == 1, got
    if rc == 0:
        assert got[1] == q
