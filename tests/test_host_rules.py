"""The library's host-side rules (tests/c/host_rules.cu, compiled with the library's own
headers and units), without a GPU."""
import os
import subprocess

import pytest

from paper_1008_2865_gb300 import build as lbbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# the library's units that hold a rule (resident_plan, pair_tiles), and what they call
UNITS = [os.path.join(lbbuild.BUILDDIR, u) for u in ("lb_resident.o", "lb_pair.o", "lb_trace.o")]


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    lbbuild.build()
    exe = str(tmp_path_factory.mktemp("rules") / "host_rules")
    subprocess.run([lbbuild._nvcc(), *lbbuild.ARCH, "-std=c++17", "-I" + lbbuild.INCLUDE,
                    "-I" + lbbuild.CSRC, os.path.join(ROOT, "tests", "c", "host_rules.cu"),
                    *UNITS, "-o", exe],
                   check=True)
    return exe


@pytest.mark.parametrize("check", ["wait_limit", "shared_launches", "swaps"])
def test_host_rule(rules, check):
    r = subprocess.run([rules, check], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
