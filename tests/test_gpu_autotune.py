"""The launch-shape autotuner times the storages whose kernels take a block size, and
no others: kernels with a CTA shape of their own would leave noise in the tuning file,
and need no scratch copy of the links."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import torch
import paper_1310_7087_gb300 as q
torch.zeros(1, device="cuda")
for group, Ns, Nt, precision in ((3, 4, 4, 0), (3, 20, 8, 0), (3, 16, 4, 1), (2, 16, 8, 0), (3, 24, 6, 1), (2, 4, 4, 1), (2, 20, 6, 0)):
    lat = q.Lattice(group, Ns, Nt, 2.3, 0, precision, q.QCD_HOT, 1)
    lat.sweep(1, 1)
    assert q.qcd_get_block(lat.h) in (64, 128, 256, 512)
    lat.close()
"""


def test_tuned_shapes(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1310_7087_gb300 import build
    build.build()
    cache = tmp_path / "tune"
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = {k: v for k, v in os.environ.items() if k != "QCD_AUTOTUNE"}
    subprocess.run([sys.executable, "-c", PROGRAM], check=True, cwd=root, timeout=300,
                   env=dict(env, QCD_AUTOTUNE_CACHE=str(cache), PYTHONPATH=root))
    tuned = sorted("_".join(line.split("_")[:3]) for line in cache.read_text().splitlines())
    assert tuned == ["su2_p0_20x6", "su2_p1_4x4", "su3_p1_24x6"], tuned
