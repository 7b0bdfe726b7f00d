"""The named ranges of nq_total_ex's host phases, as a timeline profiler gets them
(nvtx_ranges.c). Without a GPU the call ends at its pinned staging memory, with the
set counted."""
import os
import subprocess
import sys

import pytest

from paper_2511_12009_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def injection(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("nvtx") / "ranges.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    subprocess.run(["gcc", "-shared", "-fPIC", "-I", cuda, os.path.join(HERE, "nvtx_ranges.c"),
                    "-o", so], check=True)
    return so


ALL = ["nq.enumerate.count", "nq.enumerate.write", "nq.upload"]


@pytest.mark.parametrize("layout,names", [
    ("default", ALL[:1]), pytest.param("default", ALL, marks=pytest.mark.gpu),
    ("regm", ALL[:1]), pytest.param("regm", ALL, marks=pytest.mark.gpu)])
def test_total_opens_its_ranges(injection, layout, names):
    code = ("from paper_2511_12009_gb300 import nq\n"
            f"try: nq.total_ex(12, nq.make_config({layout!r}))\n"
            f"except nq.NQError as e: assert {len(names)} == 1 and e.code == nq.NQ_ENOMEM")
    r = subprocess.run([sys.executable, "-c", code], cwd=os.path.dirname(HERE),
                       env=dict(os.environ, NVTX_INJECTION64_PATH=injection), capture_output=True,
                       text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-2000:]
    seen = [line.split()[1] for line in r.stderr.splitlines() if line.startswith("range nq.")]
    assert list(dict.fromkeys(seen))[:len(names)] == names
