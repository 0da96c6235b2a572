"""The plan of small chains and stars where a cluster of 16 CTAs has no room, on a
fake of the CUDA runtime (no GPU): one cluster launch where it fits, the four
launches where the device has no such cluster or the launch is refused."""
import json
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

CHILD = """
import ctypes, json, sys
from paper_1905_13376_gb300 import binding as B
lib, fake = B.load(), ctypes.CDLL(sys.argv[1])
n, kind = int(sys.argv[2]), sys.argv[3]
h, size = ctypes.c_void_p(), ctypes.c_size_t()
assert lib.mwj_create(ctypes.byref(h), None) == 0
rel = [B.mwj_rel(0x10000 * (2 * k + 1), 0x10000 * (2 * k + 2), n) for k in range(4)]
out = B.mwj_out()
out.mode, out.total = B.MODES["count"], 0x900000
if kind == "chain":
    assert lib.mwj_join4_workspace_size(h, *rel, None, out.mode, ctypes.byref(size)) == 0
    st = lib.mwj_join4_linear(h, *rel, None, ctypes.byref(out), 0x10000000, size.value, None)
else:
    k = B.MWJ_STAR if kind == "star" else B.MWJ_LINEAR
    assert lib.mwj_workspace_size(h, k, *rel[:3], None, out.mode, ctypes.byref(size)) == 0
    join = lib.mwj_join3_star if kind == "star" else lib.mwj_join3_linear
    st = join(h, *rel[:3], None, ctypes.byref(out), 0x10000000, size.value, None)
sizes, m = (ctypes.c_uint * 256)(), ctypes.c_uint()
refused = fake.fake_launches(sizes, ctypes.byref(m))
print(json.dumps([st, lib.mwj_stream_status(h, None), list(sizes[:m.value]), refused]))
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_1905_13376_gb300 import build
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", f"-I{CUDA}/include", os.path.join(HERE, "fake_cudart.c"), "-o", so],
                   check=True)
    return so


def run(fake, n, kind, fits, launches):
    env = dict(os.environ, LD_PRELOAD=fake, FAKE_FITS=str(fits), FAKE_LAUNCHES=str(launches), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD, fake, str(n), kind], env=env, capture_output=True, text=True, cwd=ROOT)
    assert r.returncode == 0, r.stderr
    return json.loads(r.stdout.splitlines()[-1])


@pytest.mark.parametrize("kind,launches", [("linear", 4), ("star", 4), ("chain", 5)])
def test_where_the_cluster_has_no_room(fake, kind, launches):
    assert run(fake, 1 << 14, kind, 16, 16) == [0, 0, [16], 0]
    assert run(fake, 5000, kind, 8, 8) == [0, 0, [8], 0]
    assert run(fake, 1 << 14, kind, 8, 8) == [0, 0, [1] * launches, 0]
    assert run(fake, 1 << 14, kind, 1, 1) == [0, 0, [1] * launches, 0]
    # the device has room, the stream's part of it has not
    assert run(fake, 1 << 14, kind, 16, 8) == [0, 0, [1] * launches, 1]
    assert run(fake, (1 << 14) + 1, kind, 16, 16) == [0, 0, [1] * launches, 0]
