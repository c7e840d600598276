"""The three forms of the adjoint -- every step's state from level 1 (small batches), the noise
hand-off, the noise drawn again -- on the same batches: the same bits, and each against the oracle.

Batches of at most 32,768 trajectories take the first form unless ABP_ADJ_STATE_BYTES = 0, so the
paired kernels of the other two, which large batches run, are asked for by name here (tests/
test_host_adjoint.py checks which kernels each setting launches)."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_1104_2499_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FORMS = {"states": {}, "handoff": {"ABP_ADJ_STATE_BYTES": "0"}, "redraw": {"ABP_ADJ_STATE_BYTES": "0",
                                                                         "ABP_ADJ_HANDOFF_BYTES": "0"}}


@pytest.fixture(scope="module")
def abp():
    from paper_1104_2499_gb300 import abp as A
    from paper_1104_2499_gb300 import build as B

    B.build()
    A.lib()
    return A


@pytest.fixture
def form(monkeypatch):
    def use(name):
        for k in ("ABP_ADJ_STATE_BYTES", "ABP_ADJ_HANDOFF_BYTES"):
            monkeypatch.delenv(k, raising=False)
        for k, v in FORMS[name].items():
            monkeypatch.setenv(k, v)

    return use


def grads(abp, w, window=0, **kw):
    with abp.Ensemble(w, **kw) as ens:
        ens.run()
        return ens.backward(host=True, window=window).numpy(), ens.traj_grad(host=True).numpy()


def same_bits(abp, form, w, windows=(0,), **kw):
    out = {}
    for name in FORMS:
        form(name)
        out[name] = [a for window in windows for a in grads(abp, w, window, **kw)]
    for name in ("handoff", "redraw"):
        for a, b in zip(out[name], out["states"]):
            np.testing.assert_array_equal(a, b, err_msg=name)
    assert all(np.all(np.isfinite(a)) for a in out["states"])
    return out["states"]


SETS = [W.params(D=0.05), W.params(D=0.2, q=2.0, asym=0.1, gamma0=1.5), W.params(D=0.1, F0=0.3, c=0.3, d=0.7)]


# odd sizes (a thread with one trajectory); step counts with a partial last chunk and a short last
# segment; 1, 2 or 4 trajectories per thread in the forward: 1, 2 or 4 adjoint blocks per tile
@pytest.mark.parametrize("K,window,ppt", [(64, 0, 2), (256, 512, 2), (1000, 0, 2), (256, 0, 1), (256, 512, 4)])
def test_long_segments(abp, form, K, window, ppt):
    w = W.Workload(name="long", sets=SETS, n_traj=[1000, 257, 3], n_steps=[2051, 1900, 1024], dt=1e-3, seed=37,
                   v0_mode=1, checkpoint_every=K)
    same_bits(abp, form, w, (window,), schedule=1, particles_per_thread=ppt)


# one step per segment; inside one chunk; segments that mix partial and whole chunks (12, 50, 77,
# 333); multiples of 8; longer than every run
@pytest.mark.parametrize("K", [1, 3, 8, 12, 50, 64, 77, 333, 2000])
def test_segments_of_any_length(abp, form, K):
    w = W.Workload(name="chunks", sets=SETS, n_traj=[300, 65, 1], n_steps=[503, 164, 7], dt=1e-3, seed=21, v0_mode=1,
                   checkpoint_every=K)
    got = same_bits(abp, form, w, (0, 2 * K))[1]
    # another K only regroups the FP32 partial sums (the states and lambda are the same bits): at
    # most 503 additions, each off by 6e-8 of a partial sum, 3e-5 of the largest one in all
    form("states")
    ref = grads(abp, dataclasses.replace(w, checkpoint_every=64))[1]
    assert np.all(np.abs(got - ref) <= 1e-4 * np.abs(ref).max(axis=0))


# a pair of trajectories whose global ids lie on both sides of a multiple of 2^32
@pytest.mark.parametrize("name", list(FORMS))
@pytest.mark.parametrize("K", [64, 50])
def test_pair_astride_matches_its_shards(abp, form, K, name):
    form(name)
    M, cut = 700, 301

    def traj(m, base):
        w = W.Workload(name="astride", sets=[W.params(D=0.2)], n_traj=[m], n_steps=[203], dt=1e-3, seed=5, v0_mode=1,
                       checkpoint_every=K)
        return grads(abp, w, traj_base=base, particles_per_thread=2)[1]

    np.testing.assert_array_equal(traj(M, (1 << 32) - cut), np.concatenate([traj(cut, (1 << 32) - cut),
                                                                            traj(M - cut, 1 << 32)]))


# every trajectory's derivative against the oracle's FP64 tangent, over 1,000 steps where the FP32
# and FP64 paths stay together: within 1e-3 of the component or of its root mean square in the set
@pytest.mark.parametrize("name", list(FORMS))
@pytest.mark.parametrize("K,window", [(250, 0), (64, 0), (250, 500)])
def test_trajectories_match_the_oracle(abp, form, K, window, name):
    form(name)
    w = W.Workload(name="adj_traj", sets=SETS, n_traj=[1000, 513, 700], n_steps=[1000, 1000, 750], dt=1e-3, seed=35,
                   v0_mode=1, checkpoint_every=K)
    g, dv = grads(abp, w, window)
    base = w.traj_base()
    for i, p in enumerate(w.sets):
        ref = O.run_set(p, seed=w.seed, dt=w.dt, n_traj=w.n_traj[i], n_steps=w.n_steps[i], traj_base=base[i],
                        v0_mode=1, want_traj_grad=True, grad_window=window)["dvbar"]
        mine = dv[base[i]:base[i] + w.n_traj[i]]
        assert np.all(np.abs(mine - ref) <= 1e-3 * np.maximum(np.abs(ref), np.sqrt(np.mean(ref**2, axis=0)))), i
        np.testing.assert_allclose(mine.mean(axis=0), g[i], rtol=1e-9, atol=1e-12 * np.abs(g[i]).max())


# Two groups of tiles (as many blocks of the paired sweep as SMs and more than two launches): 93
# tiles of 512, odd and ragged, twice on one context, against the same trajectories set by set,
# which run as one group.  The hand-off for all (one group), for one and for two segments at a time
# (8 slots of 8 steps, 2 blocks of noise each, in 93 x 2 kernel blocks) and not at all.
SEGMENT = 2 * 16 * 93 * 2 * 8 * 2 * 2 * 128


@pytest.mark.parametrize("handoff", ["", str(SEGMENT + 4096), str(2 * SEGMENT + 4096), "0"],
                         ids=["all", "one", "two", "none"])
@pytest.mark.parametrize("K,window", [(50, 0), (50, 100), (64, 0)])
def test_two_groups_match_one(abp, form, monkeypatch, K, window, handoff):
    form("handoff")
    if handoff:
        monkeypatch.setenv("ABP_ADJ_HANDOFF_BYTES", handoff)
    n_traj, n_steps = [20001, 13003, 300, 12301, 1], [203, 200, 64, 131, 7]
    sets = SETS + [W.params(D=0.4), W.params(D=0.3, q=0.5)]
    kw = dict(particles_per_thread=2, schedule=1)
    w = W.Workload(name="groups", sets=sets, n_traj=n_traj, n_steps=n_steps, dt=1e-3, seed=39, v0_mode=1,
                   checkpoint_every=K)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with abp.Ensemble(w, **kw) as ens:
        ens.run()
        assert ens.tiles()["tiles"] == 93 and 93 * 2 >= sms
        runs = [(ens.backward(host=True, window=window).numpy(), ens.traj_grad(host=True).numpy()) for _ in range(2)]
    parts = []
    for i, b in enumerate(w.traj_base()):
        one = dataclasses.replace(w, sets=sets[i:i + 1], n_traj=n_traj[i:i + 1], n_steps=n_steps[i:i + 1])
        parts.append(grads(abp, one, window, traj_base=b, **kw))
    for g, t in runs:
        np.testing.assert_array_equal(t, np.concatenate([p[1] for p in parts]))
        np.testing.assert_array_equal(g, np.concatenate([p[0] for p in parts]))
