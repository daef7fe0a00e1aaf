"""L2 priorities of the generic passes (host code of dwt_pass.cuh, compiled into a
probe; no GPU): in every form of call the first pass reads its input and the last
pass writes its results as lines that go first, and what lies between is kept."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0808_0487_gb300", "csrc")

_PROBE = r"""
#include <stdio.h>
#include "dwt_pass.cuh"
using namespace dwt;
int main() {
    // q passes of one digit each, p = 3
    PassPlan pp[4];
    dwt_plan_s plan[4];
    std::vector<GroupJob> jobs;
    std::vector<const PassPlan*> pps;
    for (int q = 1; q <= 3; ++q) {
        pp[q].q = q;
        long long S = 1;
        for (int t = 0; t < q; ++t, S *= 3) pp[q].g[t] = PassGeom{t, 1, S, 3, 1, 0, S, 10 * q + t};
        plan[q].p = 3, plan[q].m = q, plan[q].N = S;
        jobs.push_back(GroupJob{&plan[q], nullptr, nullptr, 2, S, S});
        pps.push_back(&pp[q]);
    }
    for (int t = 0; t < 3; ++t) {
        const GroupLaunch l = group_launch<3, float2>(jobs, pps, t, true);
        for (const GroupPass& g : l.h)
            printf("grouped %d %d %d %d %d\n", t, (int)g.ntile, g.a.in_first, g.a.out_first, g.a.do_scale);
    }
    for (int q = 1; q <= 3; ++q) {
        const PassArgs a = mid_pass_args(3, 3, 8, pp[q], nullptr, nullptr, plan[q].N);
        printf("top %d %d %d\n", q, a.in_first, a.out_first);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    from paper_0808_0487_gb300 import build
    if not (os.path.exists(build.NVCC) or shutil.which(build.NVCC)):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("hints")
    (d / "probe.cu").write_text(_PROBE)
    r = subprocess.run([build.NVCC] + build.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC, "-I",
                        os.path.join(CSRC, "..", "..", "include"), str(d / "probe.cu"), "-o", str(d / "probe")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return subprocess.run([str(d / "probe")], capture_output=True, text=True, check=True).stdout.splitlines()


def test_grouped_passes(lines):
    got = [tuple(map(int, x.split()[1:])) for x in lines if x.startswith("grouped")]
    # pass t of the job with q passes (10 q + t tiles here): input first in the first and last
    # pass, output first (and the scale) in the last
    want = [(t, 10 * q + t, int(t == 0 or t == q - 1), int(t == q - 1), int(t == q - 1))
            for t in range(3) for q in range(t + 1, 4)]
    assert got == want


def test_interpolation_top_pass(lines):
    # the only pass reads samples and writes results; between two others it keeps both
    assert [x for x in lines if x.startswith("top")] == ["top 1 1 1", "top 2 0 0", "top 3 0 0"]
