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


@pytest.mark.parametrize("heads,kv,hd,max_len", [(32, 8, 128, 8192), (16, 4, 64, 2048), (8, 1, 64, 100000)])
def test_attention_workspace_grows_with_the_batch(run, heads, kv, hd, max_len):
    run(f"grows((b, L.wq_attn_workspace_bytes(b, {heads}, {kv}, {hd}, {max_len})) for b in range(1, 1200))")


@pytest.mark.parametrize("d,inter,heads,kv,hd,max_len", [(2560, 9728, 32, 8, 128, 8192), (512, 896, 8, 1, 64, 100000),
                                                         (1024, 1024, 32, 8, 128, 32768)])
def test_decoder_workspace_grows_with_the_batch(run, d, inter, heads, kv, hd, max_len):
    run(f"""
mlp = wq._MLPLayer(q({inter}, {d}, 128, 2), q({inter}, {d}, 128, 2), q({d}, {inter}, 128, 4), None, None, None, 0, 1.0)
layer = wq._DecoderLayer(q({(heads + 2 * kv) * hd}, {d}, 128, 4), q({d}, {heads * hd}, 64, 4), mlp, {heads}, {kv}, {hd}, 1e6)
grows((b, L.wq_decoder_workspace_bytes(b, ctypes.byref(layer), {max_len})) for b in range(1, 300))
""")


@pytest.mark.parametrize("d,inter,experts,top_k,group", [(4096, 4096, 8, 2, 128), (2880, 2880, 32, 4, 64),
                                                         (2048, 1024, 16, 4, 64)])
def test_moe_workspace_grows_with_the_tokens(run, d, inter, experts, top_k, group):
    run(f"""
gu, dn = q({experts * inter}, {d}, {group}, 2), q({experts * d}, {inter}, {group}, 4)
layer = wq._MoELayer(wq._MLPLayer(gu, gu, dn, 256, 256, 256, 16, 1.0), {experts}, {top_k})
for flags in (0, wq.WQ_PRENORM):
    grows((m, L.wq_moe_workspace_bytes(m, ctypes.byref(layer), flags)) for m in range(1, 65))
""")
