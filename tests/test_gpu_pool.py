"""The constant parameter pool takes the systems it took when a system's
parameters were laid out 16 bytes apart less strictly (up to 5 % smaller)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# in a process of its own, so that no other test's systems are in the pool
CODE = """
import numpy as np
from paper_2106_13281_gb300 import scenes as S
from paper_2106_13281_gb300.system import BraxSystem
keep = [BraxSystem(S.biped())]  # 28,432 bytes (27,440 before)
for k in range(3):              # 11,168 bytes each (11,136): 61,936 in all (60,848)
    d = S.quadruped()
    d["gear"] = np.asarray(d["gear"]) * (1.0 + 0.1 * k)
    keep.append(BraxSystem(d))
"""


def test_pool_takes_a_biped_and_three_quadrupeds():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
