"""Trajectories of one thread share the head of their counter blocks, which depends on the high
word of the global trajectory id.  A tile (or an adjoint pair) astride a multiple of 2^32 must
give every trajectory the bits it has in a shard that does not cross."""
import dataclasses

import numpy as np
import pytest

from paper_1104_2499_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

M, CUT = 700, 301  # one set of 700 trajectories; the first 301 ids lie below 2^32
BASE = (1 << 32) - CUT


@pytest.fixture(scope="module")
def abp():
    from paper_1104_2499_gb300 import abp as A
    from paper_1104_2499_gb300 import build as B

    B.build()
    A.lib()
    return A


def batch(m=M, **kw):
    return W.Workload(name="astride", sets=[W.params(D=0.2)], n_traj=[m], n_steps=[203], dt=1e-3, seed=5, v0_mode=1, **kw)


def states(abp, w, **kw):
    with abp.Ensemble(w, **kw) as ens:
        ens.run()
        return {k: v.numpy() for k, v in ens.state(host=True).items()}


@pytest.mark.parametrize("schedule", [1, 2])
@pytest.mark.parametrize("ppt", [1, 2, 4])
@pytest.mark.parametrize("mode", ["em", "heun", "xorshift", "fp64"])
def test_tile_astride_matches_its_shards(abp, mode, ppt, schedule):
    w = batch(scheme=int(mode == "heun"), noise=int(mode == "xorshift"))
    kw = dict(particles_per_thread=ppt, schedule=schedule, steps_per_launch=100, state_fp64=mode == "fp64")
    whole = states(abp, w, traj_base=BASE, **kw)
    low = states(abp, dataclasses.replace(w, n_traj=[CUT]), traj_base=BASE, **kw)
    high = states(abp, dataclasses.replace(w, n_traj=[M - CUT]), traj_base=1 << 32, **kw)
    for k in whole:
        np.testing.assert_array_equal(whole[k], np.concatenate([low[k], high[k]]), err_msg=k)


@pytest.mark.parametrize("handoff", ["", "0"])
@pytest.mark.parametrize("K", [64, 50])
def test_adjoint_pair_astride_matches_its_shards(abp, monkeypatch, K, handoff):
    monkeypatch.setenv("ABP_ADJ_HANDOFF_BYTES", handoff)

    def grads(m, base):
        with abp.Ensemble(batch(m, checkpoint_every=K), traj_base=base, particles_per_thread=2) as ens:
            ens.run()
            ens.backward(host=True)
            return ens.traj_grad(host=True).numpy()

    whole = grads(M, BASE)
    np.testing.assert_array_equal(whole, np.concatenate([grads(CUT, BASE), grads(M - CUT, 1 << 32)]))
