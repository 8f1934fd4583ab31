"""The autotuner tries only knobs that the kernels of a configuration read (on
the host: vd_tune.h is plain C++)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_06408_gb300", "csrc")

PROGRAM = r"""
#include "vd_tune.h"
#include <cstdio>
#include <cstdlib>
#include <cstring>
struct Field { const char* name; int32_t vd_config::*at; };
static const Field fields[] = {
    {"cell_mode", &vd_config::cell_mode}, {"warm_start", &vd_config::warm_start},
    {"verts_per_lane", &vd_config::verts_per_lane}, {"queue_per_lane", &vd_config::queue_per_lane},
    {"leaf_size", &vd_config::leaf_size}, {"warps_per_block", &vd_config::warps_per_block},
    {"precision", &vd_config::precision}, {"counters", &vd_config::counters},
    {"traversal", &vd_config::traversal}, {"cull_mode", &vd_config::cull_mode}};
int main(int argc, char** argv) {  // large, then field=value ...
  vd_config c;
  memset(&c, 0, sizeof(c));
  c.leaf_size = 16, c.verts_per_lane = 2, c.queue_per_lane = 4, c.warps_per_block = 4;
  for (int i = 2; i < argc; i++) {
    const char* eq = strchr(argv[i], '=');
    for (const Field& f : fields)
      if (!strncmp(f.name, argv[i], eq - argv[i]) && f.name[eq - argv[i]] == 0) c.*(f.at) = atoi(eq + 1);
  }
  printf("form=%d", vd::tune_form(c));
  for (int k = 0; k < vd::kTuneKnobs; k++)
    for (const vd::TuneValue& v : vd::tune_values(c, k, atoi(argv[1]) != 0))
      for (const Field& f : fields)
        if (f.at == v.field) printf(" %s=%d", f.name, v.value);
  return 0;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("tune")
    (d / "prog.cpp").write_text(PROGRAM)
    r = subprocess.run([gxx, "-std=c++17", "-Wall", "-Werror", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                        str(d / "prog.cpp"), "-o", str(d / "prog")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(large, **cfg):
        words = subprocess.run([str(d / "prog"), str(int(large)), *[f"{k}={v}" for k, v in cfg.items()]],
                               capture_output=True, text=True, check=True).stdout.split()
        return words[0], words[1:]

    return run


def test_default_kernels_read_few_knobs(plan):
    assert plan(False)[1] == ["cell_mode=1", "warps_per_block=2"]
    # 1 and 2 are the same to the large-cell pass, eight warps a block are four
    assert plan(True, warm_start=2, warps_per_block=8)[1] == [
        "cell_mode=1", "warm_start=0", "leaf_size=8", "leaf_size=32", "warps_per_block=2"]


@pytest.mark.parametrize("mode", ["precision", "counters", "traversal", "cull_mode"])
def test_the_other_modes_read_all(plan, mode):
    assert plan(False, **{mode: 1})[1] == [
        "cell_mode=1", "warm_start=1", "warm_start=2", "verts_per_lane=4", "queue_per_lane=2", "queue_per_lane=8",
        "leaf_size=8", "leaf_size=32", "warps_per_block=2", "warps_per_block=8"]


def test_thread_form_reads_the_leaf_size(plan):
    assert plan(False, cell_mode=1)[1] == ["cell_mode=0", "leaf_size=8", "leaf_size=32"]


def test_a_cached_result_holds_for_its_kernels_only(plan):
    forms = [plan(False, cull_mode=c, traversal=t, precision=p, counters=n)[0]
             for c in range(3) for t in range(2) for p in range(2) for n in range(2)]
    assert len(set(forms)) == len(forms)
