"""Words without a dense row, through every z-step kernel: a build with room for
a few rows only, in a process of its own bound to it through PULDA_LIB."""
import os
import subprocess
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import no_row_cases  # noqa: E402

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_words_without_a_row(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03581_gb300 import build
    lib = build.build(extra=[f"-DPULDA_DENSE_BYTES={no_row_cases.ROWS_BYTES}ll"], out_dir=str(tmp_path / "few_rows"))
    out = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "no_row_cases.py")], cwd=ROOT,
                         env=dict(os.environ, PULDA_LIB=lib), capture_output=True, text=True, timeout=1200)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert "all cases passed" in out.stdout
