"""Which tagged words the calls on a scratch hand over through: captured calls keep theirs, so that graphs over different scratch
cannot meet. The library's host code on a stand-in for the CUDA calls, without a GPU."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DEVICE = r"""
#include <stddef.h>
#include <string.h>
#define BASE 0x700000000000ull
int capturing = 0;
unsigned long long words = 0, counts = 0;                    /* tagged words of the last launch (0: none); last memset of 4 bytes */
static int encode(void) { return 0; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)d; *v = a == 16 ? 148 : a == 97 ? 232448 : 0; return 0; }
int cudaGetDriverEntryPoint(const char* s, void** f, unsigned long long g, int* st) { (void)s; (void)g; *f = (void*)encode; *st = 0; return 0; }
int cudaDeviceSynchronize(void) { return 0; }
int cudaStreamSynchronize(void* s) { (void)s; return 0; }
int cudaMemset(void* p, int v, size_t n) { (void)v; if (n == 4) counts = (unsigned long long)p; return 0; }
int cudaMemcpy(void* d, const void* s, size_t n, int k) { (void)s; (void)k; memset(d, 1, n); return 0; }      /* (a status word that is set) */
int cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = (void*)BASE; return 0; }
int cudaStreamIsCapturing(void* s, int* st) { (void)s; *st = capturing; return 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
int cudaLaunchKernelExC(const void* cfg, const void* f, void** args) {
    (void)cfg; (void)f;
    words = 0;
    for (int i = 0; i < 224; i += 8) {                       /* (the layer kernel's last parameter) */
        unsigned long long v;
        memcpy(&v, (char*)args[2] + i, 8);
        if (v >= BASE && v < BASE + (64ull << 20)) words = v;
    }
    return 0;
}
"""
CALLS = r"""
import ctypes, sys
lib, dev = ctypes.CDLL(sys.argv[1]), ctypes.CDLL(sys.argv[2])
capturing, words, counts = ctypes.c_int.in_dll(dev, "capturing"), ctypes.c_ulonglong.in_dll(dev, "words"), ctypes.c_ulonglong.in_dll(dev, "counts")
P = ctypes.c_void_p
def scratch(i): assert lib.chunkkv_set_workspace(P((i + 1) << 32), ctypes.c_size_t(1 << 30)) == 0
def call(captured=False):
    capturing.value = int(captured)
    st = lib.chunkkv_compress_layer(P(1 << 50), P(2 << 50), P(3 << 50), 2048, 8, 2, 64, 16, 10, 256, None, P(4 << 50), P(5 << 50), P(6 << 50), None)
    assert st == 0, st
    return words.value
"""


def run(tmp_path, code):
    from paper_2502_00299_b200 import build
    build.build()
    (tmp_path / "device.c").write_text(DEVICE)
    so = str(tmp_path / "device.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", so, str(tmp_path / "device.c")], check=True)
    r = subprocess.run([sys.executable, "-c", CALLS + code, build.LIB_PATH, so], env={**os.environ, "LD_PRELOAD": so}, cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-800:]


def test_captured_calls_keep_their_words(tmp_path):
    run(tmp_path, """
scratch(0); a = call(); assert a and call() == a
scratch(1); assert call() == a                       # nothing was captured on the first: the device was idle in between
assert call(captured=True) == a and call() == a
scratch(2); b = call(); assert b and b != a          # the second's graph may run at any time
scratch(1); assert call() == a
scratch(2); assert call(captured=True) == b
scratch(3); c = call(); assert c not in (0, a, b)
assert lib.chunkkv_device_status(None) == -6 and counts.value == c + 4      # an abandoned wait: the count of this scratch's words is cleared
""")


def test_beyond_the_last_set_of_words(tmp_path):
    run(tmp_path, """
seen = []
for i in range(8):
    scratch(i); seen.append(call(captured=True))
assert 0 not in seen and len(set(seen)) == 8
scratch(8); assert call() == 0 and call(captured=True) == 0      # by counters
scratch(3); assert call() == seen[3]
""")
