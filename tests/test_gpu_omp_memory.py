"""OMP at sides 32 and 64 keeps a factor for each leaf in flight: where another
owner of device memory leaves too little for all of them, it takes fewer leaves
at a time, with the same result.  In a process of its own, since the factors'
memory is kept from call to call."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import numpy as np, torch
from paper_2605_09190_gb300 import aqmp, synthetic
plane = torch.from_numpy(synthetic.gradient_scene(640, 1024, seed=8)).cuda()      # 160 leaves of side 64
def encode(num, den):
    code = aqmp.aqmp_encode_planes([plane], 4.0, omp=True, min_block=64, max_block=64, cap_num=num, cap_den=den)
    got = [np.copy(x) for x in code.copy()]
    code.free()
    return got
encode(1, 64)                               # everything but the factors of up to 1024 atoms
free = torch.cuda.mem_get_info()[0]
room = 700 << 20
held = torch.empty(free - room, dtype=torch.uint8, device="cuda")
sms = torch.cuda.get_device_properties(0).multi_processor_count
assert torch.cuda.mem_get_info()[0] < min(sms, 160) * 1024 * 1025 * 8
few = encode(1, 4)
again = encode(1, 4)
del held
torch.cuda.empty_cache()
all_at_once = encode(1, 4)
for a, b, c in zip(few, again, all_at_once):
    assert a.tobytes() == b.tobytes() == c.tobytes()
assert torch.cuda.mem_get_info()[0] < free - min(sms, 160) * 1024 * 1025 * 8 + (64 << 20)
print("same", len(few[0]), len(few[1]))
"""


def test_fewer_leaves_in_flight_where_memory_is_short():
    from paper_2605_09190_gb300 import build_lib
    build_lib.build()
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.startswith("same 160 ")
