"""What a build does after its sort gave up waiting (VD_ERR_TIMEOUT), on the
host: the arrays then hold anything but a permutation, and the step after the
sort must read and write in range, leave the later kernels a valid order, and
make no cell. No GPU is needed: the step's code is compiled for the host."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "vd_bvh.cu"
#include <cstdio>
#include <vector>
using namespace vd;
int main(int argc, char** argv) {
  const int n = 40, nsets = atoi(argv[1]);
  const bool failed = atoi(argv[2]) != 0, weighted = nsets > 1;
  const int shift = nsets > 1 ? 54 : 63;
  std::vector<SetInfo> sets(nsets);
  for (int s = 0; s < nsets; s++) {
    sets[s].first = n * s / nsets;
    sets[s].count = n * (s + 1) / nsets - sets[s].first;
    sets[s].weighted = s & 1;
  }
  std::vector<float> xyz(3 * n), w(n);
  for (int i = 0; i < n; i++) {
    for (int k = 0; k < 3; k++) xyz[3 * i + k] = (float)((i / 2 * 7 + k * 3) % 23) / 23.f;  // pairs of one position
    w[i] = (float)(i % 3);
  }
  std::vector<int> perm(n), inv(n, -7);
  std::vector<uint64_t> keys(n);
  for (int k = 0; k < n; k++) {
    // what passes that stopped half way leave: an older build's numbers, the same ones twice, set ids past the last
    perm[k] = failed ? (k % 2 ? 1 << 30 : -k - 1) : k;
    keys[k] = failed ? ~0ull - k : ((uint64_t)find_set(sets.data(), nsets, k) << shift) + k / 2;
  }
  std::vector<float4> sites(n);
  std::vector<unsigned char> loser(n, 9);
  for (int k = 0; k < n; k++)
    gather_site(xyz.data(), weighted ? w.data() : nullptr, perm.data(), n, sets.data(), keys.data(), shift, nsets, failed,
                sites.data(), inv.data(), loser.data(), k);
  for (int k = 0; k < n; k++)
    printf("%d %d %d %d %d %.9g %.9g\n", perm[k], inv[k], (int)loser[k], nsets > 1 ? (int)(keys[k] >> shift) : 0,
           k ? keys[k - 1] <= keys[k] : 1, sites[k].x - xyz[3 * k], sites[k].w);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2605_06408_gb300 import build

    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("sort")
    src, exe = d / "prog.cu", d / "prog"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-I", build.CSRC, "-I", os.path.join(ROOT, "include"), str(src),
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return str(exe)


@pytest.mark.parametrize("nsets", [1, 3])
@pytest.mark.parametrize("failed", [0, 1])
def test_order_after_the_sort(program, nsets, failed):
    out = subprocess.run([program, str(nsets), str(failed)], capture_output=True, text=True)
    assert out.returncode == 0
    rows = [line.split() for line in out.stdout.splitlines()]
    n = 40
    assert len(rows) == n
    bounds = [n * s // nsets for s in range(nsets + 1)]
    for k, (perm, inv, loser, s, ascending, dx, w) in enumerate(rows):
        mine = next(q for q in range(nsets) if bounds[q] <= k < bounds[q + 1])
        assert (int(perm), int(inv)) == (k, k) and int(s) == mine and int(ascending) == 1
        assert float(dx) == 0.0 and float(w) == (k % 3 if mine & 1 else 0)
        if failed:
            assert int(loser) == 1
        else:  # of two sites at one position in one set, the larger weight, then the lower index, stays
            other = k ^ 1
            alone = not (bounds[mine] <= other < bounds[mine + 1])
            mw, ow = (k % 3, other % 3) if mine & 1 else (0, 0)
            assert int(loser) == (0 if alone else int(ow > mw or (ow == mw and other < k)))
