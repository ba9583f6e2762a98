"""More suites on the bounds-checked build of the library (see
test_gpu_checked.py): builds at the edges of their tiles, hub windows at the
widths that fit, half CTAs, and the packed edge words."""
import os
import re
import subprocess
import sys

import pytest

from paper_2609_21848_gb300 import buildlib

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SUITES = ["tests/test_gpu_build.py", "tests/test_gpu_half_ctas.py", "tests/test_gpu_edge_words.py",
          "tests/test_gpu_allocator.py"]


def test_build_and_sweep_suites_on_the_checked_build():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    env = dict(os.environ, DBBC_LIBRARY=buildlib.build_checked())
    # (the no-allocation case of the half CTAs compares times, which checks change)
    r = subprocess.run([sys.executable, "-m", "pytest", *SUITES, "-m", "gpu", "-k", "not few_half_ctas", "-x", "-q",
                        "-p", "no:cacheprovider"], cwd=ROOT, env=env, capture_output=True, text=True, timeout=1200)
    tail = "\n".join((r.stdout + r.stderr).splitlines()[-30:])
    assert r.returncode == 0, tail
    m = re.search(r"(\d+) passed", tail)
    assert m and int(m.group(1)) >= 50, tail  # the suites ran, not just collected
