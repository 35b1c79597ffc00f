"""The planes per CTA of a 3D step (csrc/common.cuh, plan_zchunk), compiled for the host.

The makespan of the chunk length it picks, by playing the launch's CTAs in order onto the slots, is within 2 % of the best
of all lengths: over grids of a few columns and of many, short and long ones, for the march's pairs of planes and the
general sweep; and a plan does not depend on the one asked for before it.
"""
import heapq
import subprocess

import numpy as np
import pytest

SOURCE = r"""
#include <cstdio>
#include "common.cuh"
int main() {
  long long tiles, slots;
  int n2, per, zmax;
  double extra;
  while (std::scanf("%lld %d %lld %d %lf %d", &tiles, &n2, &slots, &per, &extra, &zmax) == 6)
    std::printf("%d\n", hydro::plan_zchunk(tiles, n2, slots, per, extra, zmax));
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    from paper_2503_04428_gb300 import build
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cu").write_text(SOURCE)
    subprocess.run([build.NVCC] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, "-cudart", "shared", str(d / "plan.cu"), "-o",
                                                              str(d / "plan")], check=True)

    def call(asked):
        text = "".join("%d %d %d %d %g %d\n" % a for a in asked)
        return [int(v) for v in subprocess.run([str(d / "plan")], input=text, capture_output=True, text=True,
                                               check=True).stdout.split()]
    return call


def _makespan(z, tiles, n2, slots, per, extra):
    chunks = -(-n2 // z)
    cost = [-(-z // per) + extra] * (tiles * (chunks - 1)) + [-(-(n2 - (chunks - 1) * z) // per) + extra] * tiles
    free = [0.0] * min(slots, len(cost))
    for c in cost:
        heapq.heapreplace(free, free[0] + c)
    return max(free)


def test_plans_are_near_the_best(plan):
    rng = np.random.default_rng(2)
    asked = [(4, 2048, 456, 1, 1.5, 2048), (1, 2000, 456, 1, 1.5, 2000), (64, 128, 152, 1, 1.5, 128),
             (6, 512, 152, 2, 1.8, 256), (171, 256, 152, 2, 1.8, 256), (4, 600, 304, 1, 1.5, 600)]
    for _ in range(40):
        tiles, n2 = int(np.exp(rng.uniform(0, np.log(300)))), int(np.exp(rng.uniform(np.log(2), np.log(900))))
        march = rng.random() < 0.5
        asked.append((tiles, n2, int(rng.choice([152, 304, 456])), 2 if march else 1, 1.8 if march else 1.5, 256 if march else n2))
    for a, z in zip(asked, plan(asked)):
        tiles, n2, slots, per, extra, zmax = a
        lengths = range(1, min(n2, zmax) + 1)
        if tiles * n2 > 20000:  # (lengths that give thousands of CTAs are never best: their starts add up)
            lengths = range(max(1, tiles * n2 // 20000), min(n2, zmax) + 1)
        best = min(_makespan(v, tiles, n2, slots, per, extra) for v in lengths)
        assert _makespan(z, tiles, n2, slots, per, extra) <= 1.02 * best, (a, z)


def test_a_plan_does_not_depend_on_the_one_before(plan):
    asked = [(64, 128, 152, 1, 1.5, 128), (64, 128, 152, 1, 40.0, 128)]
    assert plan(asked) == plan(asked[:1]) + plan(asked[1:]) == plan(asked[::-1])[::-1]
