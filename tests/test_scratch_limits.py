"""Scratch memory of the serving loop when it cannot grow: the requests at hand
fail or run one step per launch, and the server goes on.  The library runs here
without a GPU, on a stand-in for the CUDA runtime (fake_cudart.c)."""
import os
import subprocess
import sys

import pytest

from paper_1007_3109_gb300 import binding as B

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

SERVE = """
import ctypes, sys
import numpy as np
from paper_1007_3109_gb300 import binding as B
fake = ctypes.CDLL(sys.argv[1])
skip, fails = int(sys.argv[2]), int(sys.argv[3])
cfg = dict(lattice="D2Q9", nspecies=1, nx=8, ny=4, tau=[0.8], reaction="linear", kappa=0.1, precision="fp32")
rho0 = np.ones((1, 4, 8))
def status(srv, t):
    try:
        srv.result(t, 60.0)
        return B.LB_RD_OK
    except B.LbRdError as e:
        return e.status
with B.Server(1 << 30, max_slots=100, steps_per_tick=8, lattice="D2Q9", nspecies=1, precision="fp32") as srv:
    first = status(srv, srv.submit(rho0, 8, **cfg))
    fake.fake_fail_mallocs(skip, fails)
    # more requests at once than the lists of launches have places for, which end one after the other
    many = [srv.submit(rho0, 800000 + 8 * j, **cfg) for j in range(80)]
    seen = {status(srv, t) for t in many}
    left = fake.fake_fails_left()
    fake.fake_fail_mallocs(0, 0)
    last = [status(srv, srv.submit(rho0, n, **cfg)) for n in (1, 8, 13)]
    print(first, sorted(seen), left, last)
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", out, os.path.join(HERE, "fake_cudart.c")], check=True)
    return out


def _serve(fake, skip, fails):
    env = dict(os.environ, LD_PRELOAD=fake, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", SERVE, fake, str(skip), str(fails)], env=env, cwd=ROOT, timeout=300,
                       capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])
    return r.stdout.strip()


def test_served_on_the_stand_in(fake):
    assert _serve(fake, 0, 0) == f"0 [0] 0 {[0] * 3}"


def test_items_cannot_grow(fake):
    # the requests of that tick fail, the next ones are served
    out = _serve(fake, 0, 1)
    assert out.startswith("0 [") and str(B.LB_RD_ENOMEM) in out and out.endswith(f"0 {[0] * 3}")


def test_depth_descriptors_cannot_grow(fake):
    # one step per launch until they can
    assert _serve(fake, 1, 1000000).endswith(str([0] * 3))
