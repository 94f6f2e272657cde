"""A wait between the CTAs of a resident march's cluster that runs out: the run fails with a status, the
kernel ends and the context stays usable."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import sys
sys.path.insert(0, {root!r})
import paper_0906_5170_gb300 as pk, workloads as W
pk.capi.LIB_PATH = {lib!r}
c = pk.Context(0)
for p in (W.config2_piston(W.config2_heights()[0], n_harm=2, n_steps=900),
          dict(W.config2_piston(W.config2_heights()[0], n_harm=2, n_steps=900), precision="fp64"),
          W.cylinder_piston(40, [0, 1], radius=1.0, below=0.4, above=0.7, t_max=1.5, n_harm=2, precision="fp32")):
    for how in ("run", "submit"):
        try:
            pl = c.plan(p)
            pl.run() if how == "run" else pl.submit().force(-1)
        except pk.CasimirError as e:
            assert e.code == -3 and "ran out" in str(e), e
        else:
            raise AssertionError("the run did not fail: " + how)
small = W.piston_small(n_steps=300, precision="fp32")
F, per, st = c.plan(small, options={{"steps_per_launch": 3}}).run(per_sim=True)
assert abs(F[small["force_axis"]]) > 0
c.close()
"""


def test_a_wait_that_runs_out_fails_the_run(tmp_path):
    # the marches compiled with no tries at all: every wait for another CTA's rows gives up at once
    from paper_0906_5170_gb300 import build as b
    b.build()
    inc = ["-I", os.path.join(ROOT, "include"), "-I", b.CSRC]
    procs = [subprocess.Popen([b._nvcc(), *b.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", *inc, "-DRES_WAIT_TRIES=0",
                               "-c", os.path.join(b.CSRC, f), "-o", str(tmp_path / (f + ".o"))]) for f in ("res2d.cu", "rescyl.cu")]
    assert [p.wait() for p in procs] == [0, 0]
    objs = [str(tmp_path / (f + ".o")) if f in ("res2d.cu", "rescyl.cu") else os.path.join(b.OUT_DIR, f + ".o") for f in b.CU + b.CXX]
    lib = str(tmp_path / "libcasimir.so")
    subprocess.check_call([b._nvcc(), *b.ARCH, "-shared", "-o", lib, *objs, "-lpthread"])
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT, lib=lib)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout[-1000:], r.stderr[-2000:])
