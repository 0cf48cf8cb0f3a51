"""A workspace made for some number of tokens serves every smaller number.

The sizes follow launch plans for the device's SMs, so the library is loaded in a
process of its own, where two runtime queries answer for a GPU of 152 SMs.
"""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = """
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int *v, int attr, int dev) {
  (void)dev;
  *v = attr == 16 ? 152 : attr == 97 ? 232448 : 1;  /* SMs, opt-in shared memory */
  return 0;
}
"""

PRELUDE = """
import ctypes, sys
ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
from paper_2606_04238_gb300 import wq
L = wq.lib()
def grows(sizes):
    most = 0
    for m, b in sizes:
        assert b > 0, m
        assert b >= most, (m, b, most)
        most = b
q = lambda n, k, group, bits: wq._QWeight(256, 256, n, k, group, bits)
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import __graft_entry__
    __graft_entry__.build()
    d = tmp_path_factory.mktemp("fake_device")
    (d / "fake.c").write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(d / "fake.so"), str(d / "fake.c")], check=True)

    def go(code):
        r = subprocess.run([sys.executable, "-c", PRELUDE + code, str(d / "fake.so")], cwd=ROOT, capture_output=True,
                           text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
    return go


@pytest.mark.parametrize("d,inter", [(2560, 9728), (5120, 17408), (4096, 14336), (4096, 2560), (512, 896)])
def test_layer_workspace_grows_with_the_tokens(run, d, inter):
    run(f"grows((m, L.wq_workspace_bytes(m, {d}, {inter}, 16)) for m in [*range(1, 1030), *range(1030, 4200, 13), 16384])")
