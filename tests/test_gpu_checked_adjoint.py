"""The paired adjoint kernels under the checked build (ABP_DEBUG_CHECKS=1: every index checked before
the access, a violation reported as ABP_ESTATE): the noise hand-off and the noise drawn again, one
group of tiles and two, segments of whole and of partial chunks, one and several segments per launch.
No check may fail and every gradient must be the release library's bits, which must be those of the
small batches' form."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import os, sys
import numpy as np
sys.path.insert(0, os.environ["ABP_ROOT"])
from paper_1104_2499_gb300 import abp as A, workloads as W

out = {}
sets = [W.params(D=0.1), W.params(D=0.5, q=3.0, asym=0.0), W.params(D=0.02, q=0.3, gamma0=2.0, F0=0.2)]
small = dict(n_traj=[256, 100, 301], n_steps=[2000, 1900, 777])
groups = dict(n_traj=[30011, 10007, 513], n_steps=[203, 200, 64])
for tag, size, K in (("small", small, 333), ("small", small, 256), ("small", small, 500), ("small", small, 4),
                     ("groups", groups, 64), ("groups", groups, 50)):
    w = W.Workload(name="adj", sets=sets, dt=1e-3, seed=31, v0_mode=1, checkpoint_every=K, **size)
    for form, env in (("states", None), ("handoff", ""), ("redraw", "0")):
        if form == "states":
            os.environ.pop("ABP_ADJ_STATE_BYTES", None)
            os.environ.pop("ABP_ADJ_HANDOFF_BYTES", None)
        else:
            os.environ["ABP_ADJ_STATE_BYTES"] = "0"
            os.environ["ABP_ADJ_HANDOFF_BYTES"] = env
        with A.Ensemble(w, schedule=1, particles_per_thread=2) as ens:
            ens.run()
            key = "%s/%d/%s/" % (tag, K, form)
            out[key + "grad"] = ens.backward(host=True).numpy()
            out[key + "windowed"] = ens.backward(host=True, window=2 * K).numpy()
            out[key + "traj"] = ens.traj_grad(host=True).numpy()
            ens.synchronize()
np.savez(sys.argv[1], **out)
'''


def test_checked_build_runs_the_paired_adjoint_clean(tmp_path):
    from paper_1104_2499_gb300 import build as B

    libs = {"release": B.build(), "checked": B.build(extra=["-DABP_DEBUG_CHECKS=1"], out_dir=B.CHECKED_OUT)}
    outs = {}
    for name, lib in libs.items():
        path = str(tmp_path / (name + ".npz"))
        env = dict(os.environ, ABP_LIB=lib, ABP_ROOT=ROOT)
        r = subprocess.run([sys.executable, "-c", CHILD, path], env=env, capture_output=True, text=True,
                           timeout=900, cwd=ROOT)
        assert r.returncode == 0, (name, r.stderr[-4000:])
        outs[name] = np.load(path)
    assert sorted(outs["release"].files) == sorted(outs["checked"].files)
    for k in outs["release"].files:
        np.testing.assert_array_equal(outs["release"][k], outs["checked"][k], err_msg=k)
        tag, K, form, what = k.split("/")
        np.testing.assert_array_equal(outs["release"][k], outs["release"]["/".join((tag, K, "states", what))], err_msg=k)
