"""The radix sort of scan_sort.cu alone: keys of two words (which radial
statistics take when halo and distance need more than 64 bits) and of one, about
the edges of its tiles, stable, with look-backs that wait and that do not.  A
program of its own, since no entry point reaches the two-word keys at test size."""
import os
import subprocess

import pytest

from paper_2110_11408_gb300 import build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MAIN = r"""
#include "scan_sort.cu"
#include <stdio.h>
#include <numeric>
#include <random>
#include <vector>
void cso_set_error(const char*, ...) {}
int cso_sm_count() { return 152; }
thread_local long long g_cso_launches = 0;
static bool run(long long n, int bits, long long patience) {
  std::mt19937_64 rng(n * 131 + bits);
  std::vector<uint64_t> hi(n), lo(n);
  std::vector<uint32_t> val(n), want(n);
  for (long long i = 0; i < n; ++i) {
    hi[i] = bits > 64 ? rng() >> (128 - bits) : 0;
    // few distinct low words in one half, so that runs of equal keys show whether it is stable
    lo[i] = bits >= 64 ? rng() : rng() >> (64 - bits);
    if (i & 1) hi[i] &= 1, lo[i] &= 3;
    val[i] = (uint32_t)i;
  }
  std::iota(want.begin(), want.end(), 0u);
  std::stable_sort(want.begin(), want.end(), [&](uint32_t a, uint32_t b) {
    return hi[a] != hi[b] ? hi[a] < hi[b] : lo[a] < lo[b];
  });
  uint64_t *h[2], *l[2];
  uint32_t* v[2];
  for (int k = 0; k < 2; ++k)
    if (cudaMalloc((void**)&h[k], 8 * n) || cudaMalloc((void**)&l[k], 8 * n) || cudaMalloc((void**)&v[k], 4 * n)) return false;
  cudaMemcpy(h[0], hi.data(), 8 * n, cudaMemcpyHostToDevice);
  cudaMemcpy(l[0], lo.data(), 8 * n, cudaMemcpyHostToDevice);
  cudaMemcpy(v[0], val.data(), 4 * n, cudaMemcpyHostToDevice);
  Workspace ws;
  ws.cap = 64 << 20;
  ws.patience = patience;
  if (cudaMalloc((void**)&ws.base, ws.cap)) return false;
  uint64_t *ph = bits > 64 ? h[0] : nullptr, *pl = l[0];
  uint32_t* pv = v[0];
  if (radix_sort_128(&ph, &pl, &pv, bits > 64 ? h[1] : nullptr, l[1], v[1], n, bits, ws, 0) != CSO_OK) return false;
  std::vector<uint32_t> got(n);
  std::vector<uint64_t> gh(n), gl(n);
  if (cudaMemcpy(got.data(), pv, 4 * n, cudaMemcpyDeviceToHost) || cudaMemcpy(gl.data(), pl, 8 * n, cudaMemcpyDeviceToHost)) return false;
  if (bits > 64 && cudaMemcpy(gh.data(), ph, 8 * n, cudaMemcpyDeviceToHost)) return false;
  for (long long i = 0; i < n; ++i)
    if (got[i] != want[i] || gl[i] != lo[want[i]] || (bits > 64 && gh[i] != hi[want[i]])) return false;
  for (int k = 0; k < 2; ++k) cudaFree(h[k]), cudaFree(l[k]), cudaFree(v[k]);
  cudaFree(ws.base);
  return true;
}
int main() {
  int bad = 0;
  for (long long n : {2ll, 2047ll, 2048ll, 2049ll, 3072ll, 3073ll, 6145ll, 100000ll})
    for (int bits : {3, 8, 41, 64, 65, 72, 100, 128})
      for (long long patience : {LOOKBACK_PATIENCE, 0ll})
        if (!run(n, bits, patience)) printf("n %lld bits %d patience %lld\n", n, bits, patience), ++bad;
  return bad != 0;
}
"""


def test_keys_of_one_and_two_words(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, exe = str(tmp_path / "main.cu"), str(tmp_path / "main")
    with open(src, "w") as f:
        f.write(MAIN)
    subprocess.check_call([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC,
                           "-I", os.path.join(build.HERE, "..", "include"), src, "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
