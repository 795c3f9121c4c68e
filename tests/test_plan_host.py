"""CPU: the plan's rules, compiled from their header by the host compiler."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2406_12580_gb300", "csrc")


def run(tmp_path, body):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include <stdio.h>\n#include <initializer_list>\n#include "blr_plan.h"\nusing namespace blr;\nint main() {\n'
                   + body + "\n}\n")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, stdout=subprocess.PIPE, text=True).stdout


def test_teams_kept_within_a_group_walk_no_more_chains(tmp_path):
    """Rounding the teams to the channel groups never gives the busiest one another
    chain (the local order takes whole chains)."""
    out = run(tmp_path, """
  long bad = 0, rounded = 0;
  for (int io = 0; io < 2; ++io)
    for (int64_t D = 8; D <= 512; D += 8)
      for (int64_t B = 1; B < 800; ++B)
        for (int64_t L : {50, 400, 800, 1000, 2000}) {
          Plan p;
          make_plan(B, L, D, io, 1.0f, false, &p);
          if (p.seq || p.lookback) continue;
          const int64_t units = (p.n_chain + 1) / 2 * 2;
          const uint32_t all = (uint32_t)(units < kPlanTeams ? units : kPlanTeams);
          const uint32_t teams = plan_teams(p, all);
          const int64_t n_g = p.n_chain / p.B;
          rounded += teams != all;
          if (teams < 1 || teams > all || (teams != all && teams % n_g != 0) ||
              (p.n_chain + teams - 1) / teams != (p.n_chain + all - 1) / all)
            ++bad;
        }
  printf("%ld %d", bad, rounded > 0);
""")
    assert out == "0 1"
