"""The report of timeout flags that were fetched together: every family whose
flag is set is cleared and named, so that none is left to be reported by a
later call.  Host code, compiled here with stand-ins for the device flags."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2303_08953_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "sg_timeouts.h"
// device flags a b c -> message, then the flags that are left
int main(int, char** v) {
  int device[3], host[3];
  for (int k = 0; k < 3; ++k) device[k] = host[k] = std::atoi(v[1 + k]);
  const char* const names[3] = {"A", "B", "C"};
  const std::string who = sg::collect_timeouts(host, names, 3, [&](int k) { device[k] = 0; });
  std::printf("%s|%d%d%d\n", who.c_str(), device[0], device[1], device[2]);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("timeouts")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", f"-I{CSRC}", str(d / "main.cpp"), "-o", str(d / "main")],
                   check=True)
    return str(d / "main")


@pytest.mark.parametrize("flags,who", [("000", ""), ("100", "A"), ("010", "B"), ("011", "B, C"),
                                       ("101", "A, C"), ("111", "A, B, C")])
def test_every_set_flag_is_cleared_and_named(program, flags, who):
    out = subprocess.run([program, *flags], check=True, capture_output=True, text=True).stdout
    assert out.strip() == f"{who}|000"


def test_the_solver_reports_through_it():
    src = open(os.path.join(CSRC, "sg_solver.cpp")).read()
    body = src[src.index("auto report_errors"):]
    body = body[:body.index("\n  };")]
    assert "collect_timeouts(" in body and body.count("throw") == 1
