"""A batch's tuning file that an earlier build wrote, whose variant numbers stood for other tiles, is not used."""
import os
import struct
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import synthetic_inputs as si
from paper_1912_02018_gb300 import Batch
c = si.cylinder_case(96, 48, 12.0, Re=100.0, superheat_Tc=0.05)
b = Batch([c, c])
v = b.tune(2)
print("variant", v, "steps", b.domain(0).info()["steps"])
"""


def _fnv(h, data):
    for x in data:
        h = ((h ^ x) * 1099511628211) & (2 ** 64 - 1)
    return h


def test_choices_of_other_tiles_are_not_taken_over(tmp_path):
    import torch

    from paper_1912_02018_gb300 import build

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build()
    # the key without the tiles: device, precision, and of each domain the sizes, flags and cylinder
    p = torch.cuda.get_device_properties(0)
    h = _fnv(1469598103934665603, p.name.encode())
    for v in (p.major, p.minor, p.multi_processor_count, 0):
        h = _fnv(h, struct.pack("<i", v))
    for _ in range(2):
        h = _fnv(_fnv(h, struct.pack("<6i", 96, 48, 0, 0, 1, 1)), struct.pack("<3d", 12.0, 24.0, 24.0))
    path = tmp_path / "tune"
    path.write_text("%016x 3\n" % h)
    env = dict(os.environ, LBM_TUNE_CACHE=str(path), PYTHONPATH=ROOT)

    def run():
        r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr
        w = r.stdout.split()
        return int(w[1]), int(w[3])

    variant, steps = run()
    assert steps == 16  # timed: four variants, two rounds of two steps
    assert run() == (variant, 0)  # its own choice is taken over
