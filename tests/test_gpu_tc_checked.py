"""The tensor-core tile's pipeline and paths, under the checked build of the library.

The checked build (build.build(checked=True)) can keep a pair of CTAs' MMA warp from running for a while, with shorter
waits, and counts which parts of a product the tensor cores decided.  This test runs tests/checked_tc_cases.py
(collected only there) in a child process whose binding uses it.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tensor_core_tile_under_the_checked_build():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("this test needs a CUDA GPU")
    from paper_2409_17658_gb300 import build

    env = dict(os.environ, RD_CHECKED_LIB=build.build(checked=True))
    torch.cuda.empty_cache()
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.join(ROOT, "tests", "checked_tc_cases.py"), "-m", "gpu",
                        "-x", "-q", "-p", "no:cacheprovider"], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=600)
    tail = (r.stdout + r.stderr)[-3000:]
    assert r.returncode == 0, tail
    assert " passed" in r.stdout and "skipped" not in r.stdout, tail
