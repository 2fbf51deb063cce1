"""A tensor-core contraction whose waits gave up: its tiles are summed directly, a host-pointer call reports
FH_ETIMEOUT, and a later call that does not run on the tensor cores is not charged with it.

The library is built a second time with tiles that say so after their last wait (no wait runs out), and used in a
process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import sys
import numpy as np
import torch
import fh_inputs as fi
from paper_1807_02718_gb300 import fh as F
F.load_library(sys.argv[1])


def timed_out(call):
    try:
        call()
    except F.FHError as e:
        assert e.status == F.FH_ETIMEOUT, e
        return True
    return False


wl = fi.circle_gauss(J=64, W=15.0, N=64, n_x=300, n_T=500)
assert 2 * 64 * 300 * 500 > 1 << 24                    # past the few-outputs route
u = {}
for tc in (1, 0):
    pr = F.Problem(0, F.FH_MIXED_TF32)
    F.fh_set_tuning(pr.ctx, contract_tc=tc)
    pr.discretize(wl.curve, wl.omega, wl.N, wl.c, wl.p)
    pr.solve()
    pr.window_spectra(wl.a, wl.t0, wl.dt, wl.H)
    d_x, d_T = torch.from_numpy(np.ravel(wl.x)).cuda(), torch.from_numpy(wl.T).cuda()
    d_u = torch.zeros(300 * 500, device="cuda", dtype=torch.float64)
    for rep in range(4):                               # direct, captured, replayed
        F.fh_sample_p_dev(pr.ctx, 0, d_x, d_T, d_u)
        torch.cuda.synchronize()
        # 16 times of the resident fields, few outputs: the call before it is not this one's
        few = F.fh_resample_p(pr.ctx, 0, wl.T[:16], 300)
    u[tc] = d_u.cpu().numpy().reshape(300, 500)
    assert np.linalg.norm(few - u[tc][:, :16]) <= 1e-11 * np.linalg.norm(u[tc])
    assert timed_out(lambda: F.fh_resample_p(pr.ctx, 0, wl.T, 300)) == bool(tc)
    F.fh_sample_p_dev(pr.ctx, 0, d_x, d_T, d_u)        # a replayed sequence sets the flag as well
    assert timed_out(lambda: F.fh_synthesize(pr.ctx, np.ones((300, 64), dtype=complex), wl.T)) == bool(tc)
    for rep in range(4):
        assert timed_out(lambda: pr.sample(wl.x, wl.T)) == bool(tc), rep
    pr.sample(wl.x, wl.T[:16])
    pr.close()
assert np.linalg.norm(u[1] - u[0]) <= 1e-11 * np.linalg.norm(u[0])
print("ok")
'''


def test_contraction_that_gave_up(tmp_path):
    from paper_1807_02718_gb300 import build
    build.build()
    nvcc, lib, name = build._nvcc(), str(tmp_path / "libfh_gives_up.so"), "k_contract_tc"
    obj = str(tmp_path / (name + ".o"))
    subprocess.run([nvcc, *build.ARCH, *build.NVCC_FLAGS, "-DFH_TEST_CONTRACT_GIVES_UP", "-c",
                    os.path.join(build.CSRC, name + ".cu"), "-o", obj], check=True)
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources() if name not in s]
    subprocess.run([nvcc, *build.ARCH, "-shared", "-cudart", "static", "-o", lib, obj, *objs], check=True)
    env = dict(os.environ, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD, lib], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
