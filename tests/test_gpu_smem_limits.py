"""A kernel's dynamic shared-memory limit is one value, whatever mesh and block width a launch has.

The limit belongs to the kernel and holds for every thread of the process, so a value that followed the launch
could be lowered by a thread with a smaller mesh between another's call and its launch.  A child process with
cudaFuncSetAttribute interposed records the values that contexts of several meshes and widths set.
"""
import os
import subprocess
import sys
from collections import defaultdict

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RECORD = r"""
#include <dlfcn.h>
#include <stdio.h>
#include <stdlib.h>
typedef int (*set_t)(const void *, int, int);
int cudaFuncSetAttribute(const void *f, int attr, int value) {
    set_t real = (set_t)dlsym(dlopen("libcudart.so.13", RTLD_LAZY), "cudaFuncSetAttribute");
    const int rc = real(f, attr, value);
    FILE *out = fopen(getenv("RECORD_OUT"), "a");
    fprintf(out, "%p %d %d %d\n", f, attr, value, rc);
    fclose(out);
    return rc;
}
"""

CHILD = """
from paper_2007_14228_gb300 import inputs as I, ofks
for cells in ((8, 8, 8), (12, 10, 9), (100, 5, 6), (6, 96, 97)):
    for p in (2, 6, 17, 41, 70):
        s = I.lih().with_cells(cells).with_p(p, occ=1.0)
        m = I.make_mesh(s)
        X = I.initial_block(m.n_free, p, 1)
        for precision in ("fp64", "mixed"):
            ctx = ofks.context_for(s, m, beta=10.0, precision=precision, poisson_sep_tc=1, pcg_pc="separable")
            ctx.init_orbitals(X)
            ctx.step(1)
            ctx.close()
"""


def test_limits_do_not_follow_the_launch(tmp_path):
    from paper_2007_14228_gb300 import build
    build.build()
    src, so, out = tmp_path / "record.c", tmp_path / "record.so", tmp_path / "record.txt"
    src.write_text(RECORD)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(so), RECORD_OUT=str(out))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    limits = defaultdict(set)
    for line in out.read_text().splitlines():
        kern, attr, value, rc = line.split()
        assert rc == "0", line
        if attr == "8":                           # cudaFuncAttributeMaxDynamicSharedMemorySize
            limits[kern].add(int(value))
    assert len(limits) > 5
    assert all(len(v) == 1 for v in limits.values()), dict(limits)
