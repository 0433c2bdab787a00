"""The two-factor kernels' twiddle tables (csrc/pp_twiddles.h), compiled for the host:
the mean output energy of a transform of any compiled length is the largest not above
1 that one scale factor can bring it to."""
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_10252_gb300", "csrc")
PROGRAM = """
#include <cstdio>
#include "pp_twiddles.h"
int main() {
    int n1, n2;
    while (scanf("%d %d", &n1, &n2) == 2) {
        printf("%a", pp::reg_dft_gain(n1) + pp::reg_dft_gain(n2));
        for (const pp::Twiddle& w : pp::balanced_twiddles(n1, n2)) printf(" %a %a", w.x, w.y);
        printf("\\n");
    }
}
"""


def lengths():
    found = set()
    for name in sorted(os.listdir(CSRC)):
        if name.startswith(("pp_lines", "pp_cart_cols")):
            text = open(os.path.join(CSRC, name)).read()
            found |= {tuple(int(v) for v in m) for m in re.findall(r"X\((\d+), (\d+), (\d+)\)", text)}
    return sorted(found)


def test_mean_energy_of_every_compiled_length(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    ls = lengths()
    assert len(ls) == 60 and all(n == a * b and a <= b <= 32 for n, a, b in ls)
    out = subprocess.run([str(exe)], input="".join("%d %d\n" % l[1:] for l in ls), capture_output=True, text=True, check=True)
    for (n, a, b), line in zip(ls, out.stdout.splitlines()):
        v = [float.fromhex(t) for t in line.split()]
        reg, w = v[0], np.array(v[1:]).reshape(n, 2)
        used = (np.arange(b)[:, None] * np.arange(a)[None]).ravel()
        mean = reg + float((w[used] ** 2).sum(1).mean()) - 1.0
        # scaling moves all entries of one magnitude together, by an ulp: the mean falls
        # short of 1 by no more than the largest of those steps
        mags, inv = np.unique(np.abs(w[used]).ravel(), return_inverse=True)
        count = np.bincount(inv)
        step = 2.0 * mags * np.spacing(mags.astype(np.float32)).astype(float) * count / n
        assert -step[mags < 1.0].max() - 1e-12 <= mean <= 1e-12, (n, mean)
