"""Sizes of scratch that the library asks for, without a GPU: its host code runs on a stand-in for the CUDA calls that say what the
device is (148 SMs, 227 KB of shared memory)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DEVICE = """
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)d; *v = a == 16 ? 148 : a == 97 ? 232448 : 0; return 0; }
int cudaGetDriverEntryPoint(const char* s, void** f, unsigned long long g, int* st) { (void)s; (void)g; *f = (void*)1; *st = 0; return 0; }
"""
SIZES = """
import ctypes, sys
lib = ctypes.CDLL(sys.argv[1])
need = lib.chunkkv_model_workspace_bytes
need.restype = lib.chunkkv_workspace_bytes.restype = ctypes.c_size_t
def check(lens, Hq, Hkv, d, w, c, budget, layers, reuse):
    last, at = 0, 0
    for L in lens:
        if L < w or Hkv * L >= 1 << 23: continue       # (out of the library's limits)
        n = need(layers, L, Hq, Hkv, d, w, c, budget, reuse)
        assert n >= last, f"{last} bytes at {at} tokens, {n} at {L}: {(Hq, Hkv, d, w, c, budget, layers, reuse)}"
        assert n >= lib.chunkkv_workspace_bytes(L, Hq, Hkv, d, w, c), (L, Hq, Hkv, d, w, c)
        last, at = n, L
    assert last > 0
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2502_00299_b200 import build
    build.build()
    d = tmp_path_factory.mktemp("device")
    (d / "device.c").write_text(DEVICE)
    so = str(d / "device.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", so, str(d / "device.c")], check=True)

    def go(code):
        r = subprocess.run([sys.executable, "-c", SIZES + code, build.LIB_PATH], env={**os.environ, "LD_PRELOAD": so}, cwd=ROOT, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-600:]
    return go


@pytest.mark.parametrize("Hkv", [1, 2, 3, 4, 5, 6, 7, 8, 9, 12, 16, 32, 64, 160])
def test_model_scratch_never_shrinks_for_a_longer_sequence(run, Hkv):
    # few and many rows, chunk sizes of the persistent kernel and others; the lengths cover where a head gets one more CTA, where the
    # number of selector CTAs changes and where score_kernel's grid becomes a multiple of the heads
    run(f"""
for G, w in ((1, 1), (1, 8), (4, 8), (4, 32), (3, 64), (8, 32), (1, 200)):
    for c in (1, 5, 7, 8, 10, 16, 20, 32):
        check(sorted({{*range(1, 3000, 11), *range(3000, 60000, 59), *range(60000, 300000, 997)}}), G * {Hkv}, {Hkv}, 128, w, c, 4096, 32, 1)
for L in (20160, 14400, 11760, 10200, 5520):        # (tiles of 120 keys)
    check(range(L - 40, L + 40), {Hkv}, {Hkv}, 128, 8, 10, 4096, 32, 1)
    check(range(L - 40, L + 40), 8 * {Hkv}, {Hkv}, 64, 32, 5, 2048, 12, 2)
""")


def test_model_scratch_where_the_persistent_kernel_ends(run):
    # more kept chunks than it lists, more chunks than it counts: shorter sequences still run in it
    run("""
for c in (5, 10, 32):
    check([*range(c * 8192 - 400, c * 8192 + 400, 3), *range(c * 9000, c * 20000, 4001)], 8, 8, 128, 8, c, 10 ** 6, 32, 1)
    check([*range(c * 65535 - 400, c * 65535 + 400, 7), c * 70000], 4, 1, 64, 16, c, 4096, 8, 1)
""")
