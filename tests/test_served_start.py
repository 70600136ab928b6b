"""The served path whose first submit cannot make its pool or a slot: the error
is returned, and the next submit starts over instead of queueing for workers
that do not exist.  api.cu and served.cu are compiled for the host with the
CUDA runtime and the kernels faked (served_fakes.h)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_11408_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

MAIN = r"""
#include "served_fakes.h"
#include <string.h>
int main(int, char** argv) {
  cso_ctx* c = nullptr;
  CHECK(cso_init(&c, 0, 0, CSO_FLAG_SLOTS(3)) == CSO_OK);
  if (!strcmp(argv[1], "pool")) g_fail_pool = 1;
  if (!strcmp(argv[1], "slot")) g_fail_host = 2;  // of the second slot
  int32_t pos[3] = {0, 0, 0};
  uint64_t ids[1] = {7}, ticket = 0;
  cso_input in = {};
  in.pos = pos, in.ids = ids, in.n = 1;
  cso_params p;
  CHECK(cso_params_default(&p, 32768) == CSO_OK);
  cso_output out = {};
  int32_t done = 0;
  CHECK(cso_submit(c, &in, &p, &out, &ticket) == CSO_ERR_CUDA);
  CHECK(strstr(cso_last_error(), "made to fail"));
  for (int k = 0; k < 4; ++k) {
    const int rc = cso_submit(c, &in, &p, &out, &ticket);
    CHECK(rc == CSO_OK || rc == CSO_EAGAIN);
    CHECK(cso_poll(c, ticket, &done, 5000000) == CSO_OK && done == 1);
  }
  cso_free(c);
  return 0;
}
"""


def build_host(tmp_path, main):
    """main with api.cu and served.cu for the host; the program's path."""
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = os.path.join(str(tmp_path), "main.cpp"), os.path.join(str(tmp_path), "main")
    with open(src, "w") as f:
        f.write(main)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-x", "c++", "-I", os.path.join(CUDA, "include"), "-I", CSRC,
                           "-I", HERE, src, os.path.join(CSRC, "api.cu"), os.path.join(CSRC, "served.cu"), "-o", exe,
                           "-lpthread"])
    return exe


@pytest.mark.parametrize("failing", ["pool", "slot"])
def test_a_failed_start_is_not_kept(tmp_path, failing):
    subprocess.run([build_host(tmp_path, MAIN), failing], check=True, timeout=60)
