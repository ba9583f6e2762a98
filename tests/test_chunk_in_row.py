"""A CSR may have up to 2^32 - 2 entries (2^31 - 1 edges), so the position past a
chunk of the last rows may not fit 32 bits. Such a graph is too large for a
test; its position arithmetic is run on the host."""
import os
import subprocess

from paper_2609_21848_gb300 import buildlib

HERE = os.path.dirname(os.path.abspath(__file__))


def test_chunks_at_the_last_positions(tmp_path):
    exe = str(tmp_path / "chunk_in_row")
    r = subprocess.run([buildlib.nvcc(), *buildlib.ARCH, "-std=c++17", "--expt-relaxed-constexpr",
                        os.path.join(HERE, "chunk_in_row.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert (r.returncode, r.stdout) == (0, "0 wrong\n")
