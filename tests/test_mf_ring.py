"""The matrix-free product's stage ring (csrc/mf_plan.h) on the host: the generator groups, which wait
by phase parity for their own stages only, must each have waited for every earlier use of their slots."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_00438_gb300", "csrc")


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src = d / "plan.cpp"
    src.write_text('#include <cstdio>\n#include "mf_plan.h"\n'
                   "int main() { for (int f = 2; f <= 8; ++f) { auto p = wfq::tc::mf_plan(f); "
                   'std::printf("%d %d %d\\n", f, p.stages, p.groups); } }\n')
    exe = d / "plan"
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [tuple(int(v) for v in line.split()) for line in out.splitlines()]


def stale_reads(stages, groups, units=200):
    """Units whose group passes the wait on their slot although the slot's copy before has not
    landed, when that copy is the one that lags: a one-bit parity wait for phase k also passes in
    phase k - 1.  A group has seen the copies of its own earlier units only."""
    bad = []
    for u in range(stages, units):
        previous = u - stages
        if previous % groups != u % groups:
            bad.append(u)
    return bad


def test_every_slot_is_one_groups(plans):
    assert [f for f, _, _ in plans] == list(range(2, 9))
    for fit, stages, groups in plans:
        assert 1 <= groups <= stages <= fit
        assert stale_reads(stages, groups) == [], (fit, stages, groups)


def test_the_model_sees_the_depths_that_mix_groups():
    assert all(stale_reads(d, 4) for d in (5, 6, 7)) and not stale_reads(8, 4) and not stale_reads(7, 1)
