"""The tables through which the CTAs of a launch hand their row records on hold the launches of GPUs with more than 148 SMs too: a small
program over the launch plans, linked with the library's objects; no GPU."""
import os
import subprocess

import pytest

PROGRAM = r"""
#include "internal.h"
#include <initializer_list>
#include <stdio.h>
using namespace chunkkv;
int main() {
    long n = 0, tagged = 0;
    for (int sms : {132, 148, 152, 160, 161, 192})
        for (int Hkv : {1, 2, 3, 4, 5, 8, 16, 37, 74, 140, 148})
            for (int R : {1, 64, 96, 128, 130, 256})
                for (int L : {1, 300, 2048, 9001, 32768, 45016, 131072})
                    for (int c : {5, 8, 10, 20}) {
                        const int w = 1, C = (L - w + c - 1) / c;
                        ResidentPlan p;
                        TokenPlan t;
                        if (make_resident_plan(L, R, Hkv, 64, c, C, c * (C / 4) + w, sms, 231424, &p)) {
                            ++n;
                            const bool in = p.grid <= kExchangeCtas;
                            tagged += in;
                            if (p.grid > sms || resident_tagged(p) != in || (sms <= 160 && !in)) { printf("layer: %d of %d CTAs, %d heads\n", p.grid, sms, Hkv); return 1; }
                        }
                        if (make_token_plan(L, w, R, Hkv, 64, sms, 231424, &t)) {
                            ++n;
                            if (t.grid > kExchangeCtas || t.grid > sms || t.grid != t.cph * t.Hs || t.cph < 1) { printf("token: %d of %d CTAs, %d heads\n", t.grid, sms, Hkv); return 1; }
                        }
                    }
    printf("%ld plans, %ld tagged\n", n, tagged);
    return n > 5000 && tagged > 2000 ? 0 : 1;
}
"""


def test_records_of_every_plan_fit_their_table(tmp_path):
    from paper_2502_00299_b200 import build
    build.build()
    objs = [os.path.join(build.BUILD_DIR, f) for f in ("layer_resident.o", "token_kernel.o")]
    if not all(map(os.path.exists, objs)):
        pytest.skip("the library came built without its objects")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc())))
    src, exe = tmp_path / "plans.cpp", tmp_path / "plans"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", build.CSRC, "-isystem", os.path.join(cuda, "include"), str(src), *objs, "-L", os.path.join(cuda, "lib64"),
                    "-lcudart", "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], env={**os.environ, "LD_LIBRARY_PATH": os.path.join(cuda, "lib64")}, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
