"""The autotuner and cso_set_schedule keep the default schedule within reach:
where it is the fastest it is what the context runs afterwards, rule on giants
included.  api.cu compiled for the host, the path's times faked."""
import subprocess

from test_served_start import build_host

MAIN = r"""
#include "served_fakes.h"
static int g_fast = 16384;  // the giant bound under which the faked levels are fastest
int main() {
  cso_ctx* c = nullptr;
  CHECK(cso_init(&c, 0, 0, CSO_FLAG_BATCHED) == CSO_OK);
  CHECK(c->sched.max_giants(19) == 19);
  g_pipeline = [](cso_ctx* c) {
    c->nstages = 1;
    c->stage_name[0] = "level1";
    c->stage_ms[0] = c->sched.giant == g_fast && c->sched.small == 64 ? 1.0 : 2.0;
  };
  int32_t pos[3] = {0, 0, 0}, giant = 0, small = 0;
  uint64_t ids[1] = {7};
  cso_input in = {};
  in.pos = pos, in.ids = ids, in.n = 1;
  cso_params p;
  CHECK(cso_params_default(&p, 32768) == CSO_OK);
  cso_output out = {};
  CHECK(cso_autotune(c, &in, &p, &out, &giant, &small) == CSO_OK);
  CHECK(giant == 16384 && small == 64 && c->sched.max_giants(19) == 19);
  g_fast = 65536;
  CHECK(cso_autotune(c, &in, &p, &out, &giant, &small) == CSO_OK);
  CHECK(giant == 65536 && small == 64 && c->sched.max_giants(19) == ~0u);
  CHECK(cso_set_schedule(c, 16384, 32) == CSO_OK && c->sched.max_giants(19) == ~0u);
  CHECK(cso_set_schedule(c, 16384, 64) == CSO_OK && c->sched.max_giants(19) == 19);
  cso_free(c);
  return 0;
}
"""


def test_the_default_schedule_is_a_candidate(tmp_path):
    subprocess.run([build_host(tmp_path, MAIN)], check=True, timeout=60)
