"""Device memory that destroyed handles leave with the process."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import json
import numpy as np, torch
import paper_2506_02114_gb300 as mm
torch.cuda.init()
pos = np.array([[0.3, 0.2], [-0.7, 0.4], [0.1, -0.6]])
free, total = torch.cuda.mem_get_info()
hs = [mm.create(0.4, 0.3, 0.0, np.ones(3), pos, 1.0, 2200, fmm_order=4, img_half=(2.0, 2.0),
                ray_grid=(300, 300), big_queue_slots=1 << 27) for _ in range(3)]
taken = free - torch.cuda.mem_get_info()[0]
for h in hs:
    mm.run(h, 0)
maps = [mm.get_map_fixed(h) for h in hs]
for h in hs:
    mm.destroy(h)
left = free - torch.cuda.mem_get_info()[0]
print(json.dumps([total, taken, left, bool(maps[0].any()),
                  all(np.array_equal(maps[0], m) for m in maps)]))
"""


def test_queues_of_gigabytes_are_given_back():
    """Three queues of 5.6 GB alive at once, in a process of their own: after
    the handles are gone, other allocators find all but 1/32 of the device's
    memory again (a twentieth of that for allocation granularity)."""
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    total, taken, left, some, same = json.loads(r.stdout.splitlines()[-1])
    assert some and same and taken > 3 * 42 * (1 << 27)
    assert left <= 1.05 * total / 32
